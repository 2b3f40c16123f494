// CUDA-core GEMMs with arbitrary operand strides and a split-index output map.
//
// This is the FP64 path and the plain-FP32 path of every contraction of the
// Fig. 2(a) pattern (boundary x vectors, environment x vectors), and the
// general small-matrix product of the rSVD steps (projections, Q = Y R^-1).
//   C(m,n) = alpha * sum_k A(m,k) B(n,k) + beta * C(m,n)
//
// Two kernels: k_gemm (tiles of 64, 32 or 16 squared, the sum optionally split over
// a thread-block cluster) and k_gemm_big (FP32, 128-row tiles). pick() chooses.
#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"

namespace fpeps {
namespace {

// One thread's share of an operand tile of R rows (m or n) and BK terms: PER elements at a fixed
// stride from one pointer that advances by a k-tile (with index arithmetic in the loop the FP32
// kernel issued two instructions per FMA). Consecutive threads walk the contiguous axis; the next
// tile's elements stay in registers while the current one is used.
template <class T, int R, int BK>
struct TileLoader {
  static constexpr int PER = R * BK / 256;       // 8, 6 or 4
  static constexpr int W = 16 / sizeof(T);       // elements per 128-bit load
  static constexpr bool ROWRUN = BK % PER == 0;  // k-contiguous operand: PER consecutive terms of one row
  const T* q;       // this thread's first element of the current k-tile
  int64_t step, adv;    // between its elements; from one k-tile to the next
  int r0, k0, dr, dk;   // tile row and term of the first element, and their steps
  int rows;             // rows of the tile inside the matrix
  bool vec;
  T v[PER];
  __device__ TileLoader(const T* base, int64_t row0, int64_t nrows, int64_t sr, int64_t sk) {
    rows = (int)min((int64_t)R, nrows - row0);
    const int t = threadIdx.x;
    if (sk == 1 && ROWRUN) { r0 = t / (BK / PER); k0 = (t % (BK / PER)) * PER; dr = 0; dk = 1; }
    else if (sk == 1 || 256 % R != 0) { r0 = t / BK; k0 = t % BK; dr = 256 / BK; dk = 0; }
    else { r0 = t % R; k0 = t / R; dr = 0; dk = 256 / R; }
    q = base + (row0 + r0) * sr + k0 * sk;
    step = dr * sr + dk * sk;
    adv = BK * sk;
    vec = PER % 4 == 0 && ROWRUN && sk == 1 && (sr % W) == 0 && ((uintptr_t)base % 16) == 0;
  }
  // the k-tile with `left` terms to the end of the sum
  __device__ __forceinline__ void load(int64_t left) {
    if (left >= BK && rows == R) {
      if (vec) {
#pragma unroll
        for (int u = 0; u < PER / W; ++u) {
          if constexpr (W == 4) {
            const float4 x = __ldg((const float4*)q + u);
            v[4 * u] = x.x; v[4 * u + 1] = x.y; v[4 * u + 2] = x.z; v[4 * u + 3] = x.w;
          } else {
            const double2 x = __ldg((const double2*)q + u);
            v[2 * u] = x.x; v[2 * u + 1] = x.y;
          }
        }
      } else if (ROWRUN && dk == 1 && step == 1) {
#pragma unroll
        for (int u = 0; u < PER; ++u) v[u] = __ldg(q + u);
      } else {
        const T* p = q;
#pragma unroll
        for (int u = 0; u < PER; ++u, p += step) v[u] = __ldg(p);
      }
    } else {
#pragma unroll
      for (int u = 0; u < PER; ++u) v[u] = (r0 + u * dr < rows && k0 + u * dk < left) ? __ldg(q + u * step) : T(0);
    }
    q += adv;
  }
  template <int LD>
  __device__ __forceinline__ void store(T (*dst)[LD]) const {
    T* d = &dst[k0][r0];
    const int st = dk * LD + dr;
#pragma unroll
    for (int u = 0; u < PER; ++u) d[u * st] = v[u];
  }
};

// 256 threads, TM x TM outputs each, operand tiles double-buffered in shared memory. The K range
// is cut into gridDim.z slices, one per CTA of a cluster (1, 1, gridDim.z); the slices' partial
// tiles are added through distributed shared memory in slice order, in FP64, so the result does
// not depend on timing and needs no workspace.
// What bounds it: FP64 issues 2 FMA per cycle per SM here, so an FP64 product takes as long as
// the FMAs of the busiest SM, padding included, and FP32 products of few outputs are bound by the
// latency of one CTA's k-tiles. One 64 x 64 tile per CTA without a split left most SMs idle when
// there are few output tiles and a long sum. Measured on GB300, FP32, before -> after (the sizes
// of a row's calibration columns and closing vectors): 256 x 288 x 36864 5365 -> 214 us,
// 1 x 144 x 36864 4735 -> 54 us, 24 x 600 x 576 86 -> 10 us.
template <class T, int BM, int BK>
__global__ void __launch_bounds__(256) k_gemm(int64_t M, int64_t N, int64_t K, int64_t ks, T alpha,
                                              const T* __restrict__ A, int64_t a_m, int64_t a_k,
                                              const T* __restrict__ B, int64_t b_n, int64_t b_k, T beta,
                                              T* __restrict__ C, OutMap om, const int* skip) {
  if (skip && *skip) return;   // the same for every CTA of a cluster
  namespace cg = cooperative_groups;
  constexpr int TM = BM / 16;
  constexpr int TILE = BK * (BM + 1);
  static_assert(4 * TILE >= BM * BM, "the partial tile reuses the operand tiles");
  __shared__ T sh[4 * TILE];   // A and B tiles, two buffers each; then the CTA's partial tile
  auto As = [&](int b) { return reinterpret_cast<T(*)[BM + 1]>(sh + b * TILE); };
  auto Bs = [&](int b) { return reinterpret_cast<T(*)[BM + 1]>(sh + (2 + b) * TILE); };
  const int tid = threadIdx.x;
  const int64_t m0 = (int64_t)blockIdx.y * BM, n0 = (int64_t)blockIdx.x * BM;
  const int64_t kb = (int64_t)blockIdx.z * ks, ke = min(K, kb + ks);
  const int tr = tid / 16, tc = tid % 16;   // 16 x 16 thread grid
  T acc[TM][TM];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) acc[i][j] = T(0);
  TileLoader<T, BM, BK> la(A + kb * a_k, m0, M, a_m, a_k), lb(B + kb * b_k, n0, N, b_n, b_k);
  la.load(ke - kb);
  lb.load(ke - kb);
  la.store(As(0));
  lb.store(Bs(0));
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = kb; k0 < ke; k0 += BK) {
    const bool more = k0 + BK < ke;
    if (more) {
      la.load(ke - k0 - BK);
      lb.load(ke - k0 - BK);
    }
    T(*as)[BM + 1] = As(buf);
    T(*bs)[BM + 1] = Bs(buf);
#pragma unroll 16
    for (int kk = 0; kk < BK; ++kk) {
      T a[TM], b[TM];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = as[kk][tr + 16 * i];
#pragma unroll
      for (int j = 0; j < TM; ++j) b[j] = bs[kk][tc + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TM; ++j) acc[i][j] = fma(a[i], b[j], acc[i][j]);
    }
    if (more) {
      la.store(As(buf ^ 1));
      lb.store(Bs(buf ^ 1));
      __syncthreads();
      buf ^= 1;
    }
  }
  auto put = [&](int r, int c, T v) {
    const int64_t gm = m0 + r, gn = n0 + c;
    if (gm >= M || gn >= N) return;
    const int64_t addr = (gm / om.mdiv) * om.c0 + (gm % om.mdiv) * om.c1 + (gn / om.ndiv) * om.c2 + (gn % om.ndiv) * om.c3;
    v *= alpha;
    if (beta != T(0)) v += beta * C[addr];
    C[addr] = v;
  };
  if (gridDim.z == 1) {
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TM; ++j) put(tr + 16 * i, tc + 16 * j, acc[i][j]);
    return;
  }
  cg::cluster_group cl = cg::this_cluster();
  __syncthreads();   // every warp is done with the operand tiles
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TM; ++j) sh[(tr + 16 * i) * BM + tc + 16 * j] = acc[i][j];
  cl.sync();
  const int S = (int)gridDim.z, rank = (int)blockIdx.z;   // the cluster spans z
  for (int e = rank * 256 + tid; e < BM * BM; e += S * 256) {
    double s = 0.0;
    for (int z = 0; z < S; ++z) s += (double)cl.map_shared_rank(sh, z)[e];
    put(e / BM, e % BM, (T)s);
  }
  cl.sync();   // no CTA leaves while another reads its partial tile
}

// FP32 products of many 128-row tiles: 256 threads, 8 x (BN / 16) outputs per thread in strips of
// two (64-bit shared-memory reads without conflicts), k-tiles of 16 double-buffered in shared
// memory, the next tile's loads held in registers (128-bit where rows or columns are aligned).
// MF: the thread index runs along m first (column-major outputs store contiguous floats), else
// along n. BN = 64, 96 or 128, whichever pads N least: padded columns cost as much as real ones.
// Two FMAs per instruction halve the issue slots: with one each and index arithmetic in the loop
// the kernel was bound by instruction issue (68 % of the slots, 36864 x 266 x 266 255 us); now
// 167 us (31 TFLOP/s), and 8192 x 8192 x 2048 7.30 -> 5.20 ms (53 TFLOP/s of ~80). Split over K as
// in k_gemm.
constexpr int GB = 128, GK = 16, GS = GB + 2;   // GS: even (64-bit reads), and rows 8 apart on other banks
// two FP32 fused multiply-adds in one instruction (each rounded to nearest, as fmaf)
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long twice(float x) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(x));
  return r;
}

template <int BN, bool MF>
__global__ void __launch_bounds__(256, 2) k_gemm_big(int64_t M, int64_t N, int64_t K, int64_t ks, float alpha,
                                                     const float* __restrict__ A, int64_t a_m, int64_t a_k,
                                                     const float* __restrict__ B, int64_t b_n, int64_t b_k, float beta,
                                                     float* __restrict__ C, OutMap om, const int* skip) {
  if (skip && *skip) return;
  constexpr int TN = BN / 16;
  constexpr int ATILE = GK * GS, BTILE = GK * (BN + 2), HALF = GB / 2 * BN;
  __shared__ __align__(16) float sh[2 * (ATILE + BTILE) > HALF ? 2 * (ATILE + BTILE) : HALF];
  auto As = [&](int b) { return reinterpret_cast<float(*)[GS]>(sh + b * ATILE); };
  auto Bs = [&](int b) { return reinterpret_cast<float(*)[BN + 2]>(sh + 2 * ATILE + b * BTILE); };
  const int tid = threadIdx.x;
  const int64_t m0 = (int64_t)blockIdx.y * GB, n0 = (int64_t)blockIdx.x * BN;
  const int tf = tid % 16, ts = tid / 16;
  const int tm = MF ? tf : ts, tn = MF ? ts : tf;   // rows 2 tm + 32 s, 2 tm + 32 s + 1 (and for n)
  const int64_t kb = (int64_t)blockIdx.z * ks, ke = min(K, kb + ks);
  TileLoader<float, GB, GK> la(A + kb * a_k, m0, M, a_m, a_k);
  TileLoader<float, BN, GK> lb(B + kb * b_k, n0, N, b_n, b_k);
  unsigned long long acc[8][TN / 2];   // pairs of neighbouring columns
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = 0ull;
  la.load(ke - kb);
  lb.load(ke - kb);
  la.store(As(0));
  lb.store(Bs(0));
  __syncthreads();
  int buf = 0;
  for (int64_t k0 = kb; k0 < ke; k0 += GK) {
    const bool more = k0 + GK < ke;
    if (more) {
      la.load(ke - k0 - GK);
      lb.load(ke - k0 - GK);
    }
    const float(*as)[GS] = As(buf);
    const float(*bs)[BN + 2] = Bs(buf);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      float2 a[4];
      unsigned long long b[TN / 2];
#pragma unroll
      for (int s = 0; s < 4; ++s) a[s] = *(const float2*)&as[kk][2 * tm + 32 * s];
#pragma unroll
      for (int s = 0; s < TN / 2; ++s) b[s] = *(const unsigned long long*)&bs[kk][2 * tn + 32 * s];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned long long a2 = twice(i % 2 ? a[i / 2].y : a[i / 2].x);
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) fma2(acc[i][j], a2, b[j]);
      }
    }
    if (more) {
      la.store(As(buf ^ 1));
      lb.store(Bs(buf ^ 1));
      __syncthreads();
      buf ^= 1;
    }
  }
  auto put = [&](int64_t gm, int64_t mo, int64_t gn, float v) {
    if (gm >= M || gn >= N) return;
    const int64_t addr = mo + (gn / om.ndiv) * om.c2 + (gn % om.ndiv) * om.c3;
    v *= alpha;
    if (beta != 0.f) v += beta * C[addr];
    C[addr] = v;
  };
  auto val = [&](int i, int j) { return __uint_as_float((uint32_t)(acc[i][j / 2] >> (32 * (j % 2)))); };
  auto rowoff = [&](int64_t gm) { return (gm / om.mdiv) * om.c0 + (gm % om.mdiv) * om.c1; };
  if (gridDim.z == 1) {
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int64_t gm = m0 + 2 * tm + 32 * (i / 2) + i % 2, mo = rowoff(gm);
#pragma unroll
      for (int j = 0; j < TN; ++j) put(gm, mo, n0 + 2 * tn + 32 * (j / 2) + j % 2, val(i, j));
    }
    return;
  }
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int S = (int)gridDim.z, rank = (int)blockIdx.z;   // the cluster spans z
#pragma unroll
  for (int h = 0; h < 2; ++h) {   // rows 64 h .. 64 h + 63 of the tile
    __syncthreads();              // the operand tiles (h = 0), or this thread's sums below, are done with
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        sh[(2 * tm + 32 * (i / 2) + i % 2) * BN + 2 * tn + 32 * (j / 2) + j % 2] = val(4 * h + i, j);
    cl.sync();
    for (int e = rank * 256 + tid; e < HALF; e += S * 256) {
      double t = 0.0;
      for (int z = 0; z < S; ++z) t += (double)cl.map_shared_rank(sh, z)[e];
      const int64_t gm = m0 + 64 * h + e / BN;
      put(gm, rowoff(gm), n0 + e % BN, (float)t);
    }
    cl.sync();                    // nobody reads this half any more
  }
}

// Which kernel: the estimated cycles of the busiest SM. Every k-tile of a CTA costs at least the
// latency of its loads (~700 cycles, hidden when a few CTAs share the SM) and at least its FMAs at
// the rate the kernel reaches (per cycle and SM; FP64: the 2 of the hardware); a cluster's exchange
// costs ~3000 cycles. Clusters of up to 16 (opt-in above 8).
struct Pick {
  int kind;      // 0..2: k_gemm with 64, 32, 16; 3..5: k_gemm_big with BN = 128, 96, 64
  int split;
};
constexpr int MAX_SPLIT = 16;
Pick pick(int64_t M, int64_t N, int64_t K, bool f64, bool b_kfast) {
  constexpr double kSms = 152;
  Pick best{0, 1};
  double cost = 1e300;
  auto cdiv = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
  const int bm[6] = {64, 32, 16, GB, GB, GB}, bn[6] = {64, 32, 16, 128, 96, 64}, bk[6] = {16, 32, 64, GK, GK, GK};
  const double rate[6] = {45, 25, 10, 75, 75, 70};
  for (int t = 0; t < (f64 ? 3 : 6); ++t) {
    if (cdiv(M, bm[t]) > 65535 || (bn[t] == 96 && !b_kfast)) continue;   // 96: loads along k only
    const int64_t tiles = cdiv(M, bm[t]) * cdiv(N, bn[t]), nk = cdiv(K, bk[t]);
    const int share = t < 3 ? 4 : 2;   // CTAs that share an SM
    for (int s = 1; s <= MAX_SPLIT; s *= 2) {
      const int64_t it = cdiv(nk, s);
      if (it * (s - 1) >= nk) continue;   // every slice has a k-tile
      const double ctas = (double)tiles * s;
      const double fma = (double)bm[t] * bn[t] * bk[t] / (f64 ? 2.0 : rate[t]);
      const double c = it * std::max(700.0 * std::ceil(ctas / (kSms * share)), fma * std::ceil(ctas / kSms)) +
                       (s > 1 ? 3000.0 : 0.0);
      if (c < 0.98 * cost) { cost = c; best = Pick{t, s}; }
    }
  }
  return best;
}

template <class... KArgs, class... Args>
void launch(void (*kern)(KArgs...), dim3 grid, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 1;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = grid.z;
  cfg.attrs = at;
  cfg.numAttrs = grid.z > 1 ? 1 : 0;
  if (grid.z > 8) FP_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  FP_CUDA(cudaLaunchKernelEx(&cfg, kern, args...));
}

template <class T, int BM, int BK>
void run_tile(cudaStream_t s, int split, int64_t M, int64_t N, int64_t K, T alpha, const T* A, int64_t a_m, int64_t a_k,
              const T* B, int64_t b_n, int64_t b_k, T beta, T* C, OutMap om, const int* skip) {
  const int64_t ks = ((K + BK - 1) / BK + split - 1) / split * BK;
  launch(k_gemm<T, BM, BK>, dim3((unsigned)((N + BM - 1) / BM), (unsigned)((M + BM - 1) / BM), (unsigned)split), s, M, N, K,
         ks, alpha, A, a_m, a_k, B, b_n, b_k, beta, C, om, skip);
}

template <int BN>
void run_big(cudaStream_t s, int split, int64_t M, int64_t N, int64_t K, float alpha, const float* A, int64_t a_m,
             int64_t a_k, const float* B, int64_t b_n, int64_t b_k, float beta, float* C, OutMap om, const int* skip) {
  const int64_t ks = ((K + GK - 1) / GK + split - 1) / split * GK;
  launch(om.c1 == 1 ? k_gemm_big<BN, true> : k_gemm_big<BN, false>,
         dim3((unsigned)((N + BN - 1) / BN), (unsigned)((M + GB - 1) / GB), (unsigned)split), s, M, N, K, ks, alpha, A, a_m,
         a_k, B, b_n, b_k, beta, C, om, skip);
}

}  // namespace

template <class T>
void gemm_simt(cudaStream_t s, int64_t M, int64_t N, int64_t K, T alpha, const T* A, int64_t a_m, int64_t a_k,
               const T* B, int64_t b_n, int64_t b_k, T beta, T* C, OutMap om, const int* skip, bool record) {
  if (M <= 0 || N <= 0) return;
  FP_CHECK(om.mdiv > 0 && om.ndiv > 0, FPEPS_ERR_ARG, "gemm: bad output map");
  FP_CHECK((M + 63) / 64 <= 65535, FPEPS_ERR_UNSUPPORTED, "gemm: M too large for grid");
  ProfToken pt;
  if (record)
    pt = prof_begin(PROF_GEMM_SIMT, s, 2.0 * M * N * K, (double)sizeof(T) * ((double)M * K + (double)N * K + (double)M * N));
  const Pick p = pick(M, N, K, sizeof(T) == 8, b_k == 1);
  auto go = [&](auto run) { run(s, p.split, M, N, K, alpha, A, a_m, a_k, B, b_n, b_k, beta, C, om, skip); };
  if (p.kind == 0) go(run_tile<T, 64, 16>);
  else if (p.kind == 1) go(run_tile<T, 32, 32>);
  else if (p.kind == 2) go(run_tile<T, 16, 64>);
  else if constexpr (sizeof(T) == 4) {
    if (p.kind == 3) go(run_big<128>);
    else if (p.kind == 4) go(run_big<96>);
    else go(run_big<64>);
  }
  FP_LAUNCH();
  prof_end(pt, s);
}

template void gemm_simt<float>(cudaStream_t, int64_t, int64_t, int64_t, float, const float*, int64_t, int64_t,
                               const float*, int64_t, int64_t, float, float*, OutMap, const int*, bool);
template void gemm_simt<double>(cudaStream_t, int64_t, int64_t, int64_t, double, const double*, int64_t, int64_t,
                                const double*, int64_t, int64_t, double, double*, OutMap, const int*, bool);

}  // namespace fpeps
