// Randomized-SVD building blocks (Sec. IV; Halko et al. 2011, Example 1.6):
// the Gaussian sketch Omega, FP64 Gram matrices, Cholesky QR, norms and
// layout helpers.
//
// Gaussian sketch: Philox4x64-10 (Salmon et al., SC'11) keyed by (seed, layer)
// with counter (i >> 1, j, site | stage << 16, row | env << 16); the word pair
// (x0,x1) for even i and (x2,x3) for odd i gives u = ((x >> 11) + 0.5) 2^-53
// and z = sqrt(-2 ln u1) cos(2 pi u2) (Box-Muller). i is the flat row index of
// the sketched space in C order of its (bond, bundle) legs.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"
#include "rsqrt.cuh"

namespace fpeps {
namespace {

constexpr uint64_t PH_M0 = 0xD2E7470EE14C6C93ull, PH_M1 = 0xCA5A826395121157ull;
constexpr uint64_t PH_W0 = 0x9E3779B97F4A7C15ull, PH_W1 = 0xBB67AE8584CAA73Bull;

__device__ __forceinline__ void philox4x64(uint64_t c[4], uint64_t k0, uint64_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    uint64_t hi0 = __umul64hi(PH_M0, c[0]), lo0 = PH_M0 * c[0];
    uint64_t hi1 = __umul64hi(PH_M1, c[2]), lo1 = PH_M1 * c[2];
    uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += PH_W0; k1 += PH_W1;
  }
}

__device__ __forceinline__ double u53(uint64_t x) { return ((double)(x >> 11) + 0.5) * 0x1.0p-53; }

// memory position pos = hi * lo_dim + lo within a column; canonical flat index
// i = lo * hi_dim + hi when swap != 0, else i = pos.
template <class T>
__global__ void k_sketch(T* out, int64_t n_rows, int64_t k, int64_t ld, int64_t hi_dim, int64_t lo_dim, int swap,
                         uint64_t seed, uint64_t layer, uint64_t w2, uint64_t w3) {
  const int64_t n = n_rows * k;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t j = e / n_rows, pos = e % n_rows;
    int64_t i = swap ? (pos % lo_dim) * hi_dim + pos / lo_dim : pos;
    uint64_t c[4] = {(uint64_t)i >> 1, (uint64_t)j, w2, w3};
    philox4x64(c, seed, layer);
    uint64_t a = (i & 1) ? c[2] : c[0];
    uint64_t b = (i & 1) ? c[3] : c[1];
    double z = sqrt(-2.0 * log(u53(a))) * cospi(2.0 * u53(b));
    out[j * ld + pos] = (T)z;
  }
}

// G[i][j] += sum_r Y[i*ld + r] * Y[j*ld + r] over one row chunk; 32x32 tile per block.
template <class T>
__global__ void __launch_bounds__(256) k_gram(const T* __restrict__ Y, int64_t m, int64_t k, int64_t ld,
                                              int64_t chunk, double* G) {
  __shared__ double si[32][33];
  __shared__ double sj[32][33];
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (tj < ti) return;   // upper tiles only
  const int64_t r0 = blockIdx.z * chunk, r1 = min(m, r0 + chunk);
  const int tid = threadIdx.x;
  const int li = tid / 8, lj = (tid % 8) * 4;   // each thread: 1 row x 4 cols of the tile
  double acc[4] = {0, 0, 0, 0};
  for (int64_t rb = r0; rb < r1; rb += 32) {
    for (int e = tid; e < 32 * 32; e += 256) {
      int c = e / 32, rr = e % 32;
      int64_t r = rb + rr;
      int64_t ci = (int64_t)ti * 32 + c, cj = (int64_t)tj * 32 + c;
      si[c][rr] = (r < r1 && ci < k) ? (double)Y[ci * ld + r] : 0.0;
      sj[c][rr] = (r < r1 && cj < k) ? (double)Y[cj * ld + r] : 0.0;
    }
    __syncthreads();
#pragma unroll 8
    for (int rr = 0; rr < 32; ++rr) {
      double a = si[li][rr];
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[q] = fma(a, sj[lj + q][rr], acc[q]);
    }
    __syncthreads();
  }
  int64_t gi = (int64_t)ti * 32 + li;
  if (gi >= k) return;
  for (int q = 0; q < 4; ++q) {
    int64_t gj = (int64_t)tj * 32 + lj + q;
    if (gj >= k || gj < gi) continue;
    atomicAdd(&G[gi * k + gj], acc[q]);
  }
}

// FP64-class Gram of FP32 data on the FP32 pipes: dot products in double-float (Dekker 1971; Ogita, Rump
// and Oishi 2005). p = fl(a b) is added to hi by an error-free two-sum, s = fl(hi + p), and what s misses
// of hi + a b goes to lo: hi - (s - b'), exact, and a b - b' with b' = fl(s - hi), one FMA, which takes
// the error of the product along (8 operations instead of 10 with the product's error by itself; the
// same error against 64 bits over 912 random, one-signed, cancelling and graded terms, 1e-14 to 2e-13 of
// the sum of |a b|). Each 64x64 tile of an upper block of G is summed over one row chunk and added to G
// in FP64. Bound: the FP32 pipes. The operations run on two columns at once (f32x2), which changes no
// rounding, and the next rows arrive behind the sums: the 88 Grams of a 6x6, chi = 256 row (up to
// 36864 x 266) took 41 ms with scalar operations and loads between the sums, 30.5 ms with these, 23.9 ms
// with the shorter sum.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f2(float x, float y) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ void df_add_prod(F2 a, F2 na, F2 b, F2& hi, F2& lo) {   // na = -a
  const F2 s = add2(hi, mul2(a, b));
  const F2 bp = sub2(s, hi);
  const F2 nt = fma2(na, b, bp);
  lo = add2(lo, sub2(sub2(hi, sub2(s, bp)), nt));
  hi = s;
}

constexpr int GR = 16;   // rows of Y a step
__global__ void __launch_bounds__(256, 2) k_gram_df(const float* __restrict__ Y, int64_t m, int64_t k, int64_t ld,
                                                    int64_t chunk, double* G) {
  __shared__ __align__(16) float si[2][GR][68];
  __shared__ __align__(16) float sj[2][GR][68];
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (tj < ti) return;
  const int64_t r0 = blockIdx.z * chunk, r1 = min(m, r0 + chunk);
  const int tid = threadIdx.x;
  const int tr = tid / 16, tc = tid % 16;   // 4x4 outputs: rows 4 tr + a, cols 4 tc + b
  const F2 zero = f2(0.f, 0.f);
  F2 hi[4][2], lo[4][2];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) hi[a][b] = lo[a][b] = zero;
  // a thread loads row rr of 4 columns of either block; the next step's rows arrive behind this one's sums
  const int rr = tid % GR, c0 = tid / GR;
  const float* pi = Y + ((int64_t)ti * 64 + c0) * ld + rr;
  const float* pj = Y + ((int64_t)tj * 64 + c0) * ld + rr;
  float vi[4], vj[4];
  auto load = [&](int64_t rb) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool in = rb + rr < r1;
      vi[i] = in && (int64_t)ti * 64 + c0 + 16 * i < k ? pi[rb + 16 * i * ld] : 0.f;
      vj[i] = in && (int64_t)tj * 64 + c0 + 16 * i < k ? pj[rb + 16 * i * ld] : 0.f;
    }
  };
  load(r0);
  int st = 0;
  for (int64_t rb = r0; rb < r1; rb += GR, st ^= 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      si[st][rr][c0 + 16 * i] = vi[i];
      sj[st][rr][c0 + 16 * i] = vj[i];
    }
    __syncthreads();
    if (rb + GR < r1) load(rb + GR);
#pragma unroll 4
    for (int x = 0; x < GR; ++x) {
      const float4 a4 = *(const float4*)&si[st][x][4 * tr];
      const float4 b4 = *(const float4*)&sj[st][x][4 * tc];
      const float av[4] = {a4.x, a4.y, a4.z, a4.w};
      const F2 bv[2] = {f2(b4.x, b4.y), f2(b4.z, b4.w)};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const F2 p = f2(av[a], av[a]), n = f2(-av[a], -av[a]);
#pragma unroll
        for (int b = 0; b < 2; ++b) df_add_prod(p, n, bv[b], hi[a][b], lo[a][b]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 4; ++a) {
    int64_t gi = (int64_t)ti * 64 + 4 * tr + a;
    if (gi >= k) continue;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      int64_t gj = (int64_t)tj * 64 + 4 * tc + b;
      if (gj >= k || gj < gi) continue;
      const float2 h = unpack(hi[a][b / 2]), l = unpack(lo[a][b / 2]);
      atomicAdd(&G[gi * k + gj], b % 2 ? (double)h.y + (double)l.y : (double)h.x + (double)l.x);
    }
  }
}

// ---------------------------------------------------------------- Cholesky factor and its inverse
// G = R^T R (R upper, row-major, in place of the upper triangle of the Gram matrix G; the lower
// triangle is zero on entry and stays so) and X = R^-T (lower, row-major, zero on entry): the
// elimination runs on [G | I]. A pivot at or below tol * max diag means column j depends
// numerically on the columns before it: row j of R is set to zero (the column of Q it would give
// is zero), and with it row and column j of X. info[0] |= 1 for non-finite input.

// The elimination of the n columns of D = [A | I] (shared memory, rows of ld doubles, A in columns 0 ..
// n - 1, I in n .. 2 n - 1) by one CTA of NT threads; n <= 48. Warp 0 takes
// the next pivot's reciprocal root, a chain of FP64 latencies, while the warps of the other three
// sub-partitions update the rows below: behind their FMAs in the same FP64 pipe (a warp's FP64
// instruction occupies it for 64 cycles) the chain took twice as long. dg: the diagonal of R. Returns whether a pivot
// was not finite.
template <int NT>
__device__ __forceinline__ bool eliminate(double* D, int ld, int n, double cut, double* dg, int* bad) {
  __shared__ double y_s;
  const int tid = threadIdx.x, warp = tid / 32;
  double d = D[0];
  auto pivot = [&](int j) {
    const double y = isfinite(d) && d > cut ? rsqrt_fast(d) : 0.0;
    if (tid == 0) {
      y_s = y;
      dg[j] = d * y;
      if (!isfinite(d)) *bad = 1;
    }
  };
  if (warp == 0) pivot(0);
  __syncthreads();
  for (int j = 0; j < n; ++j) {
    // row j: columns j + 1 .. n - 1 of A and 0 .. j of the inverse
    if (tid < n) {
      const int c = tid < n - j - 1 ? j + 1 + tid : n + tid - (n - j - 1);
      D[j * ld + c] *= y_s;
    }
    __syncthreads();
    const int m = n - j - 1;
    if (warp == 0) {
      if (m > 0) {
        const double r = D[j * ld + j + 1];
        d = fma(-r, r, D[(j + 1) * ld + j + 1]);
        pivot(j + 1);
      }
    } else if (warp % 4 != 0) {
      auto upd = [&](int i, int c) {   // column c > j of A, or c <= j of the inverse
        if (c > j && (c < i || (i == j + 1 && c == i))) return;   // (the next pivot is taken above)
        const int cc = c > j ? c : n + c;
        D[i * ld + cc] = fma(-D[j * ld + i], D[j * ld + cc], D[i * ld + cc]);
      };
      const int u = (warp - 1 - warp / 4) * 32 + tid % 32, nu = NT / 4 * 3;
      if (n <= 32) {   // a fixed width: a division by n costs more than the update
        for (int e = u; e < m * 32; e += nu)
          if (e % 32 < n) upd(j + 1 + e / 32, e % 32);
      } else {
        for (int e = u; e < m * 48; e += nu)
          if (e % 48 < n) upd(j + 1 + e / 48, e % 48);
      }
    }
    __syncthreads();
  }
  return *bad != 0;
}

// k <= CH_SMALL: one CTA, everything in shared memory. Measured at k = 46: factor and inverse 70 + 38 us
// in two kernels before, 35 us now.
constexpr int CH_SMALL = 48;
__global__ void __launch_bounds__(1024) k_chol_inv_small(double* G, double* X, int k, double tol, int* info) {
  extern __shared__ double ch[];
  __shared__ double dmax_s;
  __shared__ int bad;
  const int ld = 2 * k + 1, tid = threadIdx.x;
  double* dg = ch + k * ld;
  for (int e = tid; e < k * k; e += 1024) {
    const int i = e / k, c = e % k;
    ch[i * ld + c] = c >= i ? G[e] : 0.0;
    ch[i * ld + k + c] = i == c ? 1.0 : 0.0;
  }
  if (tid == 0) bad = 0;
  __syncthreads();
  if (tid < 32) {
    double dm = 0;
    for (int i = tid; i < k; i += 32) dm = fmax(dm, ch[i * ld + i]);
    for (int o = 16; o; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
    if (tid == 0) dmax_s = dm;
  }
  __syncthreads();
  const bool nonfinite = eliminate<1024>(ch, ld, k, tol * dmax_s, dg, &bad);
  for (int e = tid; e < k * k; e += 1024) {
    const int i = e / k, c = e % k;
    if (c >= i) G[e] = c == i ? dg[i] : ch[i * ld + c];
    if (c <= i) X[e] = ch[i * ld + k + c];
  }
  if (tid == 0 && nonfinite) atomicOr(info, 1);
}

// Blocked over the whole GPU (cooperative launch, panels of 32): block 0 eliminates the diagonal block
// and its inverse in shared memory; every block multiplies its share of the panel row (of R to the
// right, of X to the left) by that inverse; every block updates its share of the rows below. FP64
// arithmetic (2 FMAs per cycle and SM) is the limit of the last two, so they take whatever order spreads
// the FMAs; the first is a chain of 32 pivots. Measured at k = 266: factor 484 us and inverse 257 us in
// two kernels before (a triangular solve and a warp per column), 284 us now.
constexpr int CH_NB = 32, CH_NT = 512;
__global__ void __launch_bounds__(CH_NT) k_chol_inv_coop(double* G, double* X, int k, double tol, int* info) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  __shared__ double D[CH_NB * (2 * CH_NB + 1)];
  __shared__ double dg[CH_NB];
  __shared__ double in[CH_NT / 32][CH_NB];
  __shared__ double dmax_s;
  __shared__ int bad;
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  if (blockIdx.x == 0) {
    if (tid == 0) bad = 0;
    if (warp == 0) {
      double dm = 0;
      for (int i = lane; i < k; i += 32) dm = fmax(dm, G[(int64_t)i * k + i]);
      for (int o = 16; o; o >>= 1) dm = fmax(dm, __shfl_xor_sync(0xffffffffu, dm, o));
      if (lane == 0) dmax_s = dm;
    }
    __syncthreads();
  }
  for (int p0 = 0; p0 < k; p0 += CH_NB) {
    const int nb = min(CH_NB, k - p0), p1 = p0 + nb;
    if (blockIdx.x == 0) {
      const int ld = 2 * nb + 1;
      for (int e = tid; e < nb * nb; e += CH_NT) {
        const int i = e / nb, c = e % nb;
        D[i * ld + c] = c >= i ? __ldcg(G + (int64_t)(p0 + i) * k + p0 + c) : 0.0;
        D[i * ld + nb + c] = i == c ? 1.0 : 0.0;
      }
      __syncthreads();
      eliminate<CH_NT>(D, ld, nb, tol * dmax_s, dg, &bad);
      for (int e = tid; e < nb * nb; e += CH_NT) {
        const int i = e / nb, c = e % nb;
        if (c >= i) G[(int64_t)(p0 + i) * k + p0 + c] = c == i ? dg[i] : D[i * ld + c];
        if (c <= i) X[(int64_t)(p0 + i) * k + p0 + c] = D[i * ld + nb + c];
      }
    }
    grid.sync();
    if (p1 == k && p0 == 0) break;
    // panel row: out_r = sum_{l <= r} L_rl in_l, one warp per column (lane r holds row r)
    for (int e = tid; e < nb * nb; e += CH_NT) D[(e / nb) * (CH_NB + 1) + e % nb] = __ldcg(X + (int64_t)(p0 + e / nb) * k + p0 + e % nb);
    __syncthreads();
    for (int c = blockIdx.x + gridDim.x * warp; c < k - nb; c += gridDim.x * (CH_NT / 32)) {
      double* col = c < p0 ? X + (int64_t)p0 * k + c : G + (int64_t)p0 * k + c + nb;
      if (lane < nb) in[warp][lane] = __ldcg(col + (int64_t)lane * k);
      __syncwarp();
      if (lane < nb) {
        double a0 = 0, a1 = 0;
        for (int l = 0; l < nb; l += 2) {
          a0 = fma(D[lane * (CH_NB + 1) + l], in[warp][l], a0);
          if (l + 1 < nb) a1 = fma(D[lane * (CH_NB + 1) + l + 1], in[warp][l + 1], a1);
        }
        col[(int64_t)lane * k] = a0 + a1;
      }
      __syncwarp();
    }
    grid.sync();
    // rows below: row i of [X | G] -= sum_l R[l][i] [X | R][l], columns 0 .. p1 - 1 of X, i .. k - 1 of G
    const int n = k - p1;
    for (int64_t e = blockIdx.x * (int64_t)CH_NT + tid; e < (int64_t)n * k; e += (int64_t)gridDim.x * CH_NT) {
      const int i = p1 + (int)(e / k), c = (int)(e % k);
      if (c >= p1 && c < i) continue;
      const double *r = G + (int64_t)p0 * k + i, *b = (c < p1 ? X : G) + (int64_t)p0 * k + c;
      double a0 = 0, a1 = 0, a2 = 0, a3 = 0;
      int l = 0;
      for (; l + 4 <= nb; l += 4) {
        a0 = fma(__ldcg(r + (int64_t)l * k), __ldcg(b + (int64_t)l * k), a0);
        a1 = fma(__ldcg(r + (int64_t)(l + 1) * k), __ldcg(b + (int64_t)(l + 1) * k), a1);
        a2 = fma(__ldcg(r + (int64_t)(l + 2) * k), __ldcg(b + (int64_t)(l + 2) * k), a2);
        a3 = fma(__ldcg(r + (int64_t)(l + 3) * k), __ldcg(b + (int64_t)(l + 3) * k), a3);
      }
      for (; l < nb; ++l) a0 = fma(__ldcg(r + (int64_t)l * k), __ldcg(b + (int64_t)l * k), a0);
      double* o = (c < p1 ? X : G) + (int64_t)i * k + c;
      *o = __ldcg(o) - ((a0 + a1) + (a2 + a3));
    }
    grid.sync();
  }
  if (blockIdx.x == 0 && tid == 0 && bad) atomicOr(info, 1);
}

template <class T, class S>
__global__ void k_convert(const S* in, T* out, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (T)in[e];
}

template <class T>
__global__ void k_sumsq(const T* x, int64_t n, double* out) {
  double s = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double v = (double)x[e];
    s = fma(v, v, s);
  }
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double ws[32];
  if (threadIdx.x % 32 == 0) ws[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x < 32) {
    s = threadIdx.x < blockDim.x / 32 ? ws[threadIdx.x] : 0.0;
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) atomicAdd(out, s);
  }
}

__global__ void k_sqrt1(double* x) { x[0] = sqrt(x[0]); }

// out[0] += sum x r, out[1] += sum r r (FP64)
template <class T>
__global__ void k_dot2(const T* x, const T* r, int64_t n, double* out) {
  double a = 0, b = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const double xv = (double)x[e], rv = (double)r[e];
    a = fma(xv, rv, a);
    b = fma(rv, rv, b);
  }
  for (int o = 16; o; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  __shared__ double wa[32], wb[32];
  if (threadIdx.x % 32 == 0) {
    wa[threadIdx.x / 32] = a;
    wb[threadIdx.x / 32] = b;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    a = threadIdx.x < blockDim.x / 32 ? wa[threadIdx.x] : 0.0;
    b = threadIdx.x < blockDim.x / 32 ? wb[threadIdx.x] : 0.0;
    for (int o = 16; o; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (threadIdx.x == 0) {
      atomicAdd(out, a);
      atomicAdd(out + 1, b);
    }
  }
}
// out[0] = out[0] / out[1] (1 when the reference is zero or the ratio is not finite)
__global__ void k_ratio(double* out) {
  const double r = out[1] > 0 ? out[0] / out[1] : 1.0;
  out[0] = (isfinite(r) && r > 0) ? r : 1.0;
}

template <class T>
__global__ void k_scale_inv(T* x, int64_t n, const double* nrm) {
  const double inv = 1.0 / nrm[0];
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    x[e] = (T)((double)x[e] * inv);
}

// dst[c * ld_dst + r] = src[r * ld_src + c] (r < rows, c < cols), zero for
// rows <= r < ld_dst: a padded transpose through 32 x 33 shared tiles.
template <class T>
__global__ void k_transpose_pad(const T* __restrict__ src, int64_t rows, int64_t cols, int64_t ld_src,
                                T* __restrict__ dst, int64_t ld_dst) {
  __shared__ T tile[32][33];
  const int64_t r0 = (int64_t)blockIdx.y * 32, c0 = (int64_t)blockIdx.x * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;   // 32 x 8
  for (int i = ty; i < 32; i += 8) {
    const int64_t r = r0 + i, c = c0 + tx;
    tile[i][tx] = (r < rows && c < cols) ? src[r * ld_src + c] : T(0);
  }
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int64_t c = c0 + i, r = r0 + tx;
    if (c < cols && r < ld_dst) dst[c * ld_dst + r] = tile[tx][i];
  }
}

// dst[c * rows + r] = (T) src[r * cols + c]
template <class T>
__global__ void k_convert_f64_t(const double* __restrict__ src, int64_t rows, int64_t cols, T* __restrict__ dst) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < rows * cols; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t c = e / rows, r = e % rows;
    dst[e] = (T)src[r * cols + c];
  }
}

template <class T>
__global__ void k_sub(T* out, const T* a, const T* b, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    out[e] = a[e] - b[e];
}

// Batches z of the transpose dst[z][c][r] = src[z][r][c] (strides sz, sr, 1 and dz, dc, 1) through 32 x 32
// tiles: both sides move whole sectors, and the indices cost a few operations a tile. Bound: memory.
// 54 M floats (500 x 500 x 216): 120 us (3.6 TB/s) for both orders; element by element 399 and 688 us
// (five 64-bit divisions an element, one side in pieces of 4 bytes).
template <class T>
__global__ void __launch_bounds__(256) k_transpose3(const T* __restrict__ src, T* __restrict__ dst, int64_t nz, int64_t nr,
                                                    int64_t nc, int64_t sz, int64_t sr, int64_t dz, int64_t dc) {
  __shared__ T tile[32][33];
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  const int64_t tc = (nc + 31) / 32, r0 = blockIdx.x / tc * 32, c0 = blockIdx.x % tc * 32;
  for (int64_t z = blockIdx.y; z < nz; z += gridDim.y) {
#pragma unroll
    for (int i = ty; i < 32; i += 8)
      if (r0 + i < nr && c0 + tx < nc) tile[i][tx] = src[z * sz + (r0 + i) * sr + c0 + tx];
    __syncthreads();
#pragma unroll
    for (int i = ty; i < 32; i += 8)
      if (c0 + i < nc && r0 + tx < nr) dst[z * dz + (c0 + i) * dc + r0 + tx] = tile[tx][i];
    __syncthreads();
  }
}

template <class T>
__global__ void k_permute3(const T* in, T* out, int64_t d0, int64_t d1, int64_t d2, int p0, int p1, int p2) {
  // out dims are (d[p0], d[p1], d[p2]); in is [d0][d1][d2]
  const int64_t n = d0 * d1 * d2;
  int64_t d[3] = {d0, d1, d2};
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t o2 = e % d[p2], o1 = (e / d[p2]) % d[p1], o0 = e / (d[p2] * d[p1]);
    int64_t idx[3];
    idx[p0] = o0; idx[p1] = o1; idx[p2] = o2;
    out[e] = in[(idx[0] * d1 + idx[1]) * d2 + idx[2]];
  }
}

template <class T>
__global__ void k_fill(T* x, int64_t n, T v) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) x[e] = v;
}

template <class T>
__global__ void k_finite(const T* x, int64_t n, int* flag) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    if (!isfinite((double)x[e])) flag[0] = 1;
}


// ---- small helpers used by the engine -------------------------------------
// s_j = +1 if sum_i w_i X(i, j) >= 0 else -1 (singular-vector sign gauge with
// fixed Gaussian weights w); one block per column
template <class T>
__global__ void k_col_signs(const T* X, int64_t m, int64_t ld, const T* w, double* sgn) {
  const int j = blockIdx.x;
  double s = 0;
  for (int64_t i = threadIdx.x; i < m; i += blockDim.x) s = fma((double)w[i], (double)X[(int64_t)j * ld + i], s);
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ double ws[32];
  if (threadIdx.x % 32 == 0) ws[threadIdx.x / 32] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int w = 0; w < (int)(blockDim.x / 32); ++w) t += ws[w];
    sgn[j] = t < 0 ? -1.0 : 1.0;
  }
}

template <class T>
__global__ void k_scale_cols(T* X, int64_t m, int n, int64_t ld, const double* sc) {
  const int64_t tot = m * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    int64_t j = e / m, i = e % m;
    X[j * ld + i] = (T)((double)X[j * ld + i] * sc[j]);
  }
}

// out(i, j) = X(i, j) * d_j + out(i, j) with d_j = R[j * k + j] (the diagonal of a
// row-major FP64 k x k matrix), one FP32 (or FP64) fused multiply-add per element
template <class T>
__global__ void k_add_diag_cols(const T* X, int64_t m, int n, int64_t ldx, const double* R, int k, T* out,
                                int64_t ldo) {
  const int64_t tot = m * n;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / m, i = e % m;
    out[j * ldo + i] = fma(X[j * ldx + i], (T)R[j * (int64_t)k + j], out[j * ldo + i]);
  }
}
// [x][x_w][x'] -> [x_w][x][x'] in every row. The order is a table in shared memory (rows of at most
// BUNDLE_MAX elements), a CTA moves nr whole rows a step: one 32-bit division an element, where four 64-bit ones paced it (54 M floats, rows
// of 216: 218 -> 72 us, 6 TB/s).
constexpr int BUNDLE_MAX = 4096;
template <class T>
__global__ void __launch_bounds__(256) k_bundle_outer(const T* __restrict__ in, T* __restrict__ out, int64_t rows, int n, int nw,
                                                      int64_t nr) {
  __shared__ unsigned from[BUNDLE_MAX];
  const unsigned B = (unsigned)(n * nw * n);
  auto source = [&](unsigned o) {
    const unsigned xp = o % n, x = o / n % n, xw = o / (n * n);
    return (x * nw + xw) * n + xp;
  };
  const bool table = B <= BUNDLE_MAX;
  if (table)
    for (unsigned o = threadIdx.x; o < B; o += 256) from[o] = source(o);
  __syncthreads();
  for (int64_t r0 = blockIdx.x * nr; r0 < rows; r0 += gridDim.x * nr) {
    const unsigned tot = (unsigned)min(nr, rows - r0) * B;
    const T* src = in + r0 * B;
    T* dst = out + r0 * B;
    for (unsigned e = threadIdx.x; e < tot; e += 256) {
      const unsigned r = e / B;
      dst[e] = src[r * B + (table ? from[e - r * B] : source(e - r * B))];
    }
  }
}
template <class T>
__global__ void k_zero_diag(T* A, int k, int64_t ld) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < k) A[j * ld + j] = T(0);
}

__global__ void k_mul_vec(const double* a, const double* b, double* out, int n) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) out[i] = a[i] * b[i];
}

__global__ void k_gather_cols(const double* V, const int* order, int k, double* out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)k * k; e += (int64_t)gridDim.x * blockDim.x) {
    int r = (int)(e / k), i = (int)(e % k);
    out[e] = V[(int64_t)order[r] * k + i];
  }
}

template <class T>
__global__ void k_set_identity(T* X, int64_t m, int n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < m * n; e += (int64_t)gridDim.x * blockDim.x)
    X[e] = (e / m == e % m) ? T(1) : T(0);
}

int grid_for(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g > 152 * 32 ? 152 * 32 : (g < 1 ? 1 : g));
}

}  // namespace

template <class T>
void gaussian_sketch(cudaStream_t s, T* out, int64_t n_rows, int64_t k, int64_t ld, const int64_t* perm_div,
                     uint64_t seed, uint64_t layer, uint64_t w2, uint64_t w3) {
  int64_t hi = perm_div ? perm_div[0] : 1, lo = perm_div ? perm_div[1] : n_rows;
  // algorithmic bytes: the n x k matrix written once (the draws are FP64 arithmetic)
  ProfToken pt = prof_begin(PROF_SKETCH, s, 0.0, (double)sizeof(T) * n_rows * k);
  k_sketch<T><<<grid_for(n_rows * k), 256, 0, s>>>(out, n_rows, k, ld, hi, lo, perm_div ? 1 : 0, seed, layer, w2, w3);
  FP_LAUNCH();
  prof_end(pt, s);
}

template <class T>
void gram_f64(cudaStream_t s, const T* Y, int64_t m, int64_t k, int64_t ld, double* G) {
  FP_CUDA(cudaMemsetAsync(G, 0, sizeof(double) * k * k, s));
  if (sizeof(T) == 4) {
    int tiles = (int)((k + 63) / 64);
    int64_t tri = (int64_t)tiles * (tiles + 1) / 2;
    int64_t nchunk = std::max<int64_t>(1, 152 * 6 / tri);   // three full waves of two CTAs an SM at most
    int64_t chunk = ((m + nchunk - 1) / nchunk + 15) / 16 * 16;
    if (chunk < 16) chunk = 16;
    nchunk = (m + chunk - 1) / chunk;
    dim3 grid(tiles, tiles, (unsigned)std::max<int64_t>(nchunk, 1));
    ProfToken pt = prof_begin(PROF_GRAM, s, 2.0 * m * k * k, 4.0 * m * k);
    k_gram_df<<<grid, 256, 0, s>>>((const float*)Y, m, k, ld, chunk, G);
    FP_LAUNCH();
    prof_end(pt, s);
    return;
  }
  int tiles = (int)((k + 31) / 32);
  int64_t target_blocks = 152 * 8;
  int64_t tri = (int64_t)tiles * (tiles + 1) / 2;
  int64_t nchunk = (target_blocks + tri - 1) / tri;
  int64_t chunk = (m + nchunk - 1) / nchunk;
  chunk = ((chunk + 31) / 32) * 32;
  if (chunk < 32) chunk = 32;
  nchunk = (m + chunk - 1) / chunk;
  if (nchunk < 1) nchunk = 1;
  dim3 grid(tiles, tiles, (unsigned)nchunk);
  ProfToken pt = prof_begin(PROF_GRAM, s, 2.0 * m * k * k, (double)sizeof(T) * m * k);
  k_gram<T><<<grid, 256, 0, s>>>(Y, m, k, ld, chunk, G);
  FP_LAUNCH();
  prof_end(pt, s);
}

void cholesky_inverse_f64(cudaStream_t s, double* G, double* X, int k, int* info) {
  FP_CHECK(k <= 1024, FPEPS_ERR_UNSUPPORTED, "cholesky: k > 1024");
  double tol = 1e-13;
  ProfToken pt = prof_begin(PROF_FACTOR, s, 2.0 * k * k * k / 3.0, 16.0 * k * k);
  FP_CUDA(cudaMemsetAsync(X, 0, sizeof(double) * k * k, s));
  if (k <= CH_SMALL) {
    k_chol_inv_small<<<1, 1024, (size_t)(k * (2 * k + 1) + k) * sizeof(double), s>>>(G, X, k, tol, info);
    FP_LAUNCH();
  } else {
    static PerContext<int> resident;
    const int max_blocks = resident.get([] {
      int dev = 0, sms = 0, per = 0;
      FP_CUDA(cudaGetDevice(&dev));
      FP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
      FP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_chol_inv_coop, CH_NT, 0));
      return sms * std::max(per, 0);
    });
    const int blocks = std::min(max_blocks, 152);
    FP_CHECK(blocks >= 1, FPEPS_ERR_CUDA, "cholesky: no co-resident blocks");
    void* args[] = {&G, &X, &k, &tol, &info};
    count_launch();
    FP_CUDA(cudaLaunchCooperativeKernel((void*)k_chol_inv_coop, blocks, CH_NT, args, 0, s));
  }
  prof_end(pt, s);
}

template <class T>
void convert_f64(cudaStream_t s, const double* in, T* out, int64_t n) {
  k_convert<T, double><<<grid_for(n), 256, 0, s>>>(in, out, n);
  FP_LAUNCH();
}
template <class T>
void to_f64(cudaStream_t s, const T* in, double* out, int64_t n) {
  k_convert<double, T><<<grid_for(n), 256, 0, s>>>(in, out, n);
  FP_LAUNCH();
}

template <class T>
void frob_norm_f64(cudaStream_t s, const T* x, int64_t n, double* out) {
  FP_CUDA(cudaMemsetAsync(out, 0, sizeof(double), s));
  k_sumsq<T><<<grid_for(n), 256, 0, s>>>(x, n, out);
  FP_LAUNCH();
  k_sqrt1<<<1, 1, 0, s>>>(out);
  FP_LAUNCH();
}

template <class T>
void scale_against(cudaStream_t s, const T* x, const T* r, int64_t n, double* out) {
  FP_CUDA(cudaMemsetAsync(out, 0, 2 * sizeof(double), s));
  k_dot2<T><<<grid_for(n), 256, 0, s>>>(x, r, n, out);
  FP_LAUNCH();
  k_ratio<<<1, 1, 0, s>>>(out);
  FP_LAUNCH();
}

template <class T>
void scale_by_inv(cudaStream_t s, T* x, int64_t n, const double* nrm) {
  k_scale_inv<T><<<grid_for(n), 256, 0, s>>>(x, n, nrm);
  FP_LAUNCH();
}

template <class T>
void sub_into(cudaStream_t s, T* out, const T* a, const T* b, int64_t n) {
  if (n <= 0) return;
  k_sub<T><<<grid_for(n), 256, 0, s>>>(out, a, b, n);
  FP_LAUNCH();
}

template <class T>
void transpose_pad(cudaStream_t s, const T* src, int64_t rows, int64_t cols, int64_t ld_src, T* dst, int64_t ld_dst) {
  if (rows <= 0 || cols <= 0) return;
  const int64_t gy = (ld_dst + 31) / 32, gx = (cols + 31) / 32;
  FP_CHECK(gy < 65536, FPEPS_ERR_UNSUPPORTED, "transpose: too many rows");
  k_transpose_pad<T><<<dim3((unsigned)gx, (unsigned)gy), dim3(32, 8), 0, s>>>(src, rows, cols, ld_src, dst, ld_dst);
  FP_LAUNCH();
}

template <class T>
void add_diag_cols(cudaStream_t s, const T* X, int64_t m, int n, int64_t ldx, const double* R, int k, T* out,
                   int64_t ldo) {
  if (m * n == 0) return;
  k_add_diag_cols<T><<<grid_for(m * n), 256, 0, s>>>(X, m, n, ldx, R, k, out, ldo);
  FP_LAUNCH();
}
template <class T>
void bundle_outer(cudaStream_t s, const T* in, T* out, int64_t rows, int n, int nw) {
  const int64_t tot = rows * n * nw * n;
  if (tot == 0) return;
  const int64_t nr = std::max<int64_t>(1, BUNDLE_MAX / ((int64_t)n * nw * n));
  k_bundle_outer<T><<<(unsigned)std::min<int64_t>((rows + nr - 1) / nr, 152 * 8), 256, 0, s>>>(in, out, rows, n, nw, nr);
  FP_LAUNCH();
}
template <class T>
void zero_diag(cudaStream_t s, T* A, int k, int64_t ld) {
  if (k <= 0) return;
  k_zero_diag<T><<<(k + 255) / 256, 256, 0, s>>>(A, k, ld);
  FP_LAUNCH();
}

template <class T>
void convert_f64_t(cudaStream_t s, const double* src, int64_t rows, int64_t cols, T* dst) {
  k_convert_f64_t<T><<<grid_for(rows * cols), 256, 0, s>>>(src, rows, cols, dst);
  FP_LAUNCH();
}

template <class T>
void permute3(cudaStream_t s, const T* in, T* out, int64_t d0, int64_t d1, int64_t d2, int p0, int p1, int p2) {
  // p2 == 2 keeps the rows and is no transpose; a side below 16 would leave most of a 32 x 32 tile empty
  const int64_t d[3] = {d0, d1, d2}, si[3] = {d1 * d2, d2, 1};
  if (p2 != 2 && d2 >= 16 && d[p2] >= 16) {
    int64_t so[3];
    so[p2] = 1;
    so[p1] = d[p2];
    so[p0] = d[p1] * d[p2];
    const int z = 1 - p2;   // the third axis
    const int64_t tiles = ((d[p2] + 31) / 32) * ((d2 + 31) / 32);
    if (tiles <= INT32_MAX) {
      const dim3 grid((unsigned)tiles, (unsigned)std::min<int64_t>(std::max<int64_t>(d[z], 1), 65535));
      k_transpose3<T><<<grid, 256, 0, s>>>(in, out, d[z], d[p2], d2, si[z], si[p2], so[z], so[2]);
      FP_LAUNCH();
      return;
    }
  }
  k_permute3<T><<<grid_for(d0 * d1 * d2), 256, 0, s>>>(in, out, d0, d1, d2, p0, p1, p2);
  FP_LAUNCH();
}

template <class T>
void fill(cudaStream_t s, T* x, int64_t n, T v) {
  if (n <= 0) return;
  k_fill<T><<<grid_for(n), 256, 0, s>>>(x, n, v);
  FP_LAUNCH();
}

template <class T>
void check_finite(cudaStream_t s, const T* x, int64_t n, int* flag) {
  if (n <= 0) return;
  k_finite<T><<<grid_for(n), 256, 0, s>>>(x, n, flag);
  FP_LAUNCH();
}


template <class T>
void col_signs(cudaStream_t s, const T* X, int64_t m, int n, int64_t ld, const T* w, double* sgn) {
  if (n <= 0) return;
  k_col_signs<T><<<n, 256, 0, s>>>(X, m, ld, w, sgn);
  FP_LAUNCH();
}
template <class T>
void scale_cols(cudaStream_t s, T* X, int64_t m, int n, int64_t ld, const double* sc) {
  if (n <= 0 || m <= 0) return;
  k_scale_cols<T><<<grid_for(m * n), 256, 0, s>>>(X, m, n, ld, sc);
  FP_LAUNCH();
}
void mul_vec(cudaStream_t s, const double* a, const double* b, double* out, int n) {
  k_mul_vec<<<(n + 255) / 256, 256, 0, s>>>(a, b, out, n);
  FP_LAUNCH();
}
void gather_cols_f64(cudaStream_t s, const double* V, const int* order, int k, double* out) {
  k_gather_cols<<<grid_for((int64_t)k * k), 256, 0, s>>>(V, order, k, out);
  FP_LAUNCH();
}
template <class T>
void set_identity(cudaStream_t s, T* X, int64_t m, int n) {
  k_set_identity<T><<<grid_for(m * n), 256, 0, s>>>(X, m, n);
  FP_LAUNCH();
}
template <class T>
void copy_cols(cudaStream_t s, const T* src, int64_t m, int n, T* dst) {
  FP_CUDA(cudaMemcpyAsync(dst, src, sizeof(T) * m * n, cudaMemcpyDeviceToDevice, s));
}

// Row selection within every column of a column-major block (charge sectors of
// the block-sparse mode): gather dst[i + j ldd] = src[idx[i] + j lds], scatter
// dst[idx[i] + j ldd] = src[i + j lds], for i < n, j < k. idx holds valid rows of
// the indexed side (checked on the host when the lists are built).
template <class T>
__global__ void k_gather_rows(const T* __restrict__ src, int64_t lds, const int64_t* __restrict__ idx, int64_t n,
                              int64_t k, T* __restrict__ dst, int64_t ldd) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * k; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / n, i = e % n;
    dst[j * ldd + i] = src[j * lds + idx[i]];
  }
}
template <class T>
__global__ void k_scatter_rows(const T* __restrict__ src, int64_t lds, const int64_t* __restrict__ idx, int64_t n,
                               int64_t k, T* __restrict__ dst, int64_t ldd) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n * k; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / n, i = e % n;
    dst[j * ldd + idx[i]] = src[j * lds + i];
  }
}
template <class T>
void gather_rows(cudaStream_t s, const T* src, int64_t lds, const int64_t* idx, int64_t n, int64_t k, T* dst,
                 int64_t ldd) {
  if (n * k == 0) return;
  k_gather_rows<T><<<grid_for(n * k), 256, 0, s>>>(src, lds, idx, n, k, dst, ldd);
  FP_LAUNCH();
}
template <class T>
void scatter_rows(cudaStream_t s, const T* src, int64_t lds, const int64_t* idx, int64_t n, int64_t k, T* dst,
                  int64_t ldd) {
  if (n * k == 0) return;
  k_scatter_rows<T><<<grid_for(n * k), 256, 0, s>>>(src, lds, idx, n, k, dst, ldd);
  FP_LAUNCH();
}

// dst (cols x rows, column-major, ld ldd) = transpose of src (rows x cols, ld lds)
template <class T>
__global__ void k_transpose_block(const T* __restrict__ src, int64_t lds, int64_t rows, int64_t cols,
                                  T* __restrict__ dst, int64_t ldd) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < rows * cols;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t j = e / rows, i = e % rows;
    dst[i * ldd + j] = src[j * lds + i];
  }
}
template <class T>
void transpose_block(cudaStream_t s, const T* src, int64_t lds, int64_t rows, int64_t cols, T* dst, int64_t ldd) {
  if (rows * cols == 0) return;
  k_transpose_block<T><<<grid_for(rows * cols), 256, 0, s>>>(src, lds, rows, cols, dst, ldd);
  FP_LAUNCH();
}

#define INST(T)                                                                                              \
  template void gaussian_sketch<T>(cudaStream_t, T*, int64_t, int64_t, int64_t, const int64_t*, uint64_t,    \
                                   uint64_t, uint64_t, uint64_t);                                            \
  template void gram_f64<T>(cudaStream_t, const T*, int64_t, int64_t, int64_t, double*);                      \
  template void convert_f64<T>(cudaStream_t, const double*, T*, int64_t);                                    \
  template void to_f64<T>(cudaStream_t, const T*, double*, int64_t);                                          \
  template void frob_norm_f64<T>(cudaStream_t, const T*, int64_t, double*);                                  \
  template void scale_by_inv<T>(cudaStream_t, T*, int64_t, const double*);                                   \
  template void scale_against<T>(cudaStream_t, const T*, const T*, int64_t, double*);                        \
  template void permute3<T>(cudaStream_t, const T*, T*, int64_t, int64_t, int64_t, int, int, int);            \
  template void transpose_pad<T>(cudaStream_t, const T*, int64_t, int64_t, int64_t, T*, int64_t);            \
  template void sub_into<T>(cudaStream_t, T*, const T*, const T*, int64_t);                                   \
  template void convert_f64_t<T>(cudaStream_t, const double*, int64_t, int64_t, T*);                         \
  template void add_diag_cols<T>(cudaStream_t, const T*, int64_t, int, int64_t, const double*, int, T*, int64_t); \
  template void zero_diag<T>(cudaStream_t, T*, int, int64_t);                                                 \
  template void bundle_outer<T>(cudaStream_t, const T*, T*, int64_t, int, int);                               \
  template void fill<T>(cudaStream_t, T*, int64_t, T);                                                        \
  template void check_finite<T>(cudaStream_t, const T*, int64_t, int*);                                      \
  template void col_signs<T>(cudaStream_t, const T*, int64_t, int, int64_t, const T*, double*);                         \
  template void scale_cols<T>(cudaStream_t, T*, int64_t, int, int64_t, const double*);                        \
  template void set_identity<T>(cudaStream_t, T*, int64_t, int);                                              \
  template void copy_cols<T>(cudaStream_t, const T*, int64_t, int, T*);                                      \
  template void gather_rows<T>(cudaStream_t, const T*, int64_t, const int64_t*, int64_t, int64_t, T*, int64_t);   \
  template void scatter_rows<T>(cudaStream_t, const T*, int64_t, const int64_t*, int64_t, int64_t, T*, int64_t); \
  template void transpose_block<T>(cudaStream_t, const T*, int64_t, int64_t, int64_t, T*, int64_t);
INST(float)
INST(double)
template void fill<int>(cudaStream_t, int*, int64_t, int);

}  // namespace fpeps
