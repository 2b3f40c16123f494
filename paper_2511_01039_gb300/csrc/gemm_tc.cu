// Split-precision tensor-core GEMM for sm_103a: tcgen05.mma with TMEM accumulators, operands
// staged in shared memory by TMA (cp.async.bulk.tensor).
//
//   C(m,n) = sum_k A[m][k] B[n][k]      A [M][lda], B [N][ldb] fp32, k contiguous
//
// This carries the two chi^2-class contractions of every Fig. 2(a) application (boundary x
// vectors, environment x vectors) and the tall-times-small products of the QR and truncation
// steps.
//
// The split. Every FP32 element is written as x 2^e = hi + lo with hi, lo FP16 (11 significant
// bits each) and one power of two 2^e per row and segment of 256 terms, chosen so that the
// segment's largest element lies in [2^14, 2^15). hi + lo then carries 22 bits of every element
// within 2^-17 of its segment's largest (|x - hi - lo| <= 2^-22 |x|, the same as a split into two
// TF32 numbers; lo is a multiple of 2^-24, so smaller ones keep 2^-39 of the largest). The product is
// a_lo b_hi + a_hi b_lo + a_hi b_hi, FP16 x FP16 being exact in the FP32 accumulator.
// The smaller ones matter where the operands are graded against each other (A falls along k where B
// rises, or A's large terms meet zeros of B): they carry the sum. Such products are found by the
// splitting pass (Grading, common.cuh) and computed again with the on-chip split.
// Why FP16 and not TF32 halves: an FP16 MMA does twice the terms of a TF32 MMA of the same cost,
// and hi and lo together take the four bytes of the FP32 element, so both operands are split
// once, in one streaming pass (k_split_planes), and the GEMM moves no more bytes than before.
// Splitting on chip (gemm_onchip.cu) repeats it in every tile that uses an operand, and its converter
// warps pace that kernel at 40 % of what three MMAs per term allow.
//
// Layout of a split operand: row-major, per k-block of 32 terms 32 hi then 32 lo (128 bytes, one
// swizzle row), so one TMA box brings both and the MMAs step through it in 32-byte strides.
//
// Accumulation: the tensor cores add into the FP32 accumulator with truncation, which drifts over
// long sums (measured ~1e-5 relative at K = 2048, ~1e-3 at K = 1e5). K is therefore cut into
// chunks of 256 terms, the scale segments; each chunk accumulates in a fresh TMEM accumulator and
// the epilogue warps add it, times both segments' 2^-e, to a running FP32 sum in registers. Two
// accumulators alternate, so the MMAs never wait for a drain.
//
// Schedule: persistent, one CTA pair per two SMs (cta_group::2, tiles of 256 rows) or, when M
// fits 128-row tiles better, one CTA per SM; tiles are BN <= 256 columns wide. Whole waves of tiles
// run one tile per pair in turn (neighbouring tiles at the same time, which share operands in
// L2); the tiles of the last, partial wave are cut into equal runs of (tile, chunk) units over all
// pairs, and the pieces of a cut tile are added by a second kernel in a fixed order.
//
// What bounds it: 3 MMAs per term at the tensor rate (631 TFLOP/s, a third of the measured BF16
// rate) for long sums, the epilogue and the power limit otherwise. Measured on GB300, splitting pass
// included, on-chip TF32 split -> this: 8192 x 8192 x 8192 4.06 -> 2.19 ms (502 TFLOP/s), 108000 x
// 9936 x 500 4.32 -> 2.38 ms, 108000 x 1728 x 500 0.79 -> 0.54 ms, 500 x 9936 x 108000 4.41 ->
// 3.66 ms (a third of it the splitting pass over 4.3 GB of B). The mainloop alone reaches 600
// TFLOP/s at K = 500. Error against FP64 on N(0,1) data 9.4e-7 (on-chip TF32 1.8e-6: an FP16 MMA
// adds twice the terms per truncating accumulation).
//
// Every wait on an mbarrier is bounded: a timeout sets an error word, the CTA stops issuing work,
// waits (bounded) for what it has in flight, frees its TMEM and exits; CTAs that start after an
// error return at once.
#include <cuda.h>
#include <cuda_fp16.h>

#include <algorithm>
#include <mutex>

#include "common.cuh"
#include "tc_ptx.cuh"

namespace fpeps {
namespace {

using namespace tc;

constexpr int BK = 32;                 // terms per k-block
constexpr int SEG = 256;               // terms per scale segment and per accumulation chunk
constexpr int CHB = SEG / BK;          // k-blocks per chunk
constexpr int ROWB = 4 * BK;           // bytes of a row's k-block: 32 hi + 32 lo
constexpr int BM = 128, BNMAX = 256;   // rows per CTA, columns per tile at most
constexpr int TILE_A = BM * ROWB;
constexpr int ACC_COLS = BNMAX;        // TMEM columns of one accumulator (two fill the 512)

// ---------------------------------------------------------------- splitting pass
struct SplitOp {
  const float* x;
  int64_t rows, ld;
  __half* planes;   // [rows][nk][64]
  float* inv;       // [nseg][rows]: 2^-e
};

// Counts of a segment for Grading, by the whole warp: its elements are src[0 .. len), largest top (finite,
// not zero). large: at least 2^-9 of it, tiny: not zero and below 2^-17.
struct Terms {
  int large, tiny;
};
__device__ __noinline__ Terms count_terms(const float* src, int len, float top) {
  const float high = 0x1p-9f * top, low = 0x1p-17f * top;
  int nl = 0, nt = 0;
  for (int i = threadIdx.x % 32; i < len; i += 32) {
    const float x = fabsf(src[i]);
    nl += x >= high;
    nt += x != 0.f && x < low;
  }
  return Terms{__reduce_add_sync(0xffffffffu, nl), __reduce_add_sync(0xffffffffu, nt)};
}

// One warp per (row, segment): 8 elements per lane, the segment's largest magnitude by shuffles,
// one read and one write of four bytes per element (HBM-bound, with two thirds of the issue slots and
// all warps of an SM in flight: 32 registers at most). An infinite or NaN element keeps its value in hi (lo
// becomes NaN), so non-finite input still gives non-finite output. The terms of a segment are counted
// only where one of them is tiny.
__global__ void __launch_bounds__(256, 8) k_split_planes(SplitOp a, SplitOp b, int64_t K, unsigned nk, unsigned nseg, Grading* gr, int mark) {
  const int lane = threadIdx.x % 32;
  const unsigned wa = (unsigned)a.rows * nseg, tot = wa + (unsigned)b.rows * nseg;   // a segment takes 1 KB: 32 bits do
  const unsigned nw = gridDim.x * (blockDim.x / 32);
  for (unsigned w = blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32; w < tot; w += nw) {
    const SplitOp& o = w < wa ? a : b;
    const unsigned v = w < wa ? w : w - wa, row = v / nseg, seg = v - row * nseg;
    const int64_t k = (int64_t)seg * SEG + lane * 8;
    const float* src = o.x + row * o.ld + k;
    float f[8];
    if (k + 8 <= K) {   // rows start on 16-byte boundaries and k is a multiple of 8
      const float4 u0 = __ldcs((const float4*)src), u1 = __ldcs((const float4*)src + 1);
      f[0] = u0.x; f[1] = u0.y; f[2] = u0.z; f[3] = u0.w;
      f[4] = u1.x; f[5] = u1.y; f[6] = u1.z; f[7] = u1.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) f[i] = k + i < K ? src[i] : 0.f;
    }
    float mx = 0.f;
    uint32_t mn = ~0u;   // smallest magnitude that is not zero, twice its bits less one
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      mx = fmaxf(mx, fabsf(f[i]));
      mn = min(mn, 2 * __float_as_uint(f[i]) - 1);
    }
    const uint32_t mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));   // largest magnitude of the segment
    const int ex = (int)(mb >> 23);
    const int e = mb == 0 || ex == 255 ? 0 : min(141 - ex, 126);
    const float sc = __int_as_float((e + 127) << 23);
    uint32_t h2[4], l2[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float x0 = f[2 * i] * sc, x1 = f[2 * i + 1] * sc;
      const __half2 h = __floats2half2_rn(x0, x1);
      const float2 hf = __half22float2(h);
      const __half2 l = __floats2half2_rn(x0 - hf.x, x1 - hf.y);
      h2[i] = *(const uint32_t*)&h;
      l2[i] = *(const uint32_t*)&l;
    }
    const unsigned kb = seg * CHB + lane / 4;
    if (kb < nk) {   // the last k-block is padded with zeros
      __half* dst = o.planes + ((int64_t)row * nk + kb) * (2 * BK) + (lane % 4) * 8;
      *(uint4*)dst = make_uint4(h2[0], h2[1], h2[2], h2[3]);
      *(uint4*)(dst + BK) = make_uint4(l2[0], l2[1], l2[2], l2[3]);
    }
    if (lane == 0) o.inv[(int64_t)seg * o.rows + row] = __int_as_float((127 - e) << 23);
    const float top = __uint_as_float(mb);
    if (__any_sync(0xffffffffu, mn < 2 * __float_as_uint(0x1p-17f * top) - 1) && mb != 0 && ex != 255) {
      const int len = (int)min((int64_t)SEG, K - (int64_t)seg * SEG);
      const Terms n = count_terms(src - lane * 8, len, top);
      if (lane == 0 && n.tiny > min(24, 2 + len / 8)) {
        gr->deep[w < wa ? 0 : 1] = mark;
        if (n.large < 3 * len / 32) gr->narrow = mark;
      }
    }
  }
}

// The second half of the test, over the FP32 operands, only when the other operand is deep
__global__ void __launch_bounds__(256) k_uneven(SplitOp a, SplitOp b, int64_t K, unsigned nseg, Grading* gr, int mark) {
  const bool need[2] = {*(volatile int*)&gr->deep[1] == mark, *(volatile int*)&gr->deep[0] == mark};
  if (!need[0] && !need[1]) return;
  const int lane = threadIdx.x % 32;
  const int64_t wa = a.rows * (int64_t)nseg, tot = wa + b.rows * (int64_t)nseg;
  for (int64_t w = blockIdx.x * (int64_t)(blockDim.x / 32) + threadIdx.x / 32; w < tot; w += (int64_t)gridDim.x * (blockDim.x / 32)) {
    const int which = w < wa ? 0 : 1;
    // voted: other warps raise the word meanwhile, and all lanes take part in the reductions below
    if (__any_sync(0xffffffffu, !need[which] || *(volatile int*)&gr->uneven[which] == mark)) continue;
    const SplitOp& o = which ? b : a;
    const int64_t v = which ? w - wa : w, row = v / nseg, seg = v % nseg;
    const int len = (int)min((int64_t)SEG, K - seg * SEG);
    const float* src = o.x + row * o.ld + seg * SEG;
    float mx = 0.f;
    for (int i = lane; i < len; i += 32) mx = fmaxf(mx, fabsf(src[i]));
    const uint32_t mb = __reduce_max_sync(0xffffffffu, __float_as_uint(mx));
    if (mb == 0 || (mb >> 23) == 255) continue;   // zeros: exact; not finite: so is the result
    const Terms n = count_terms(src, len, __uint_as_float(mb));
    if (lane == 0 && n.large < len - 1 - len / 16) gr->uneven[which] = mark;
  }
}

// ---------------------------------------------------------------- the GEMM
struct TcArgs {
  int M, N;
  int mdiv, ndiv;         // output map, addr = (m / mdiv) c0 + (m % mdiv) c1 + (n / ndiv) c2 + (n % ndiv) c3
  int64_t c0, c1, c2, c3;
  float* C;
  const float *inva, *invb;   // 2^-e of row r in chunk c at [c * stride + r]
  int64_t sca, scb;           // strides (0: one scale per row)
  float* part;            // pieces of cut tiles: [2 slots][bn][rows]
  int* err;
  int bn;                 // columns per tile (multiple of 32)
  int m_fast;             // rasterisation: 1 => consecutive tiles walk m
  int mt, nt;
  int full, ntiles;       // tiles [0, full) run whole, [full, ntiles) are cut over all slots
  int slots, uslots;      // uslots: slots that get units of the cut tiles
  int nk, nch;            // k-blocks, chunks
  int accumulate;         // C += instead of C =
  int hold;               // self-test of the bounded waits: issue no loads, so every consumer times out
};

// The work of one slot (CTA pair or CTA) in order: whole tiles, then its run of units.
struct Work {
  int tile, c0, c1;
};
struct WorkIter {
  int t, u, u1;   // next whole tile; next and last unit of the cut tiles
  __device__ WorkIter(const TcArgs& g, int slot) {
    const int64_t U = (int64_t)(g.ntiles - g.full) * g.nch;
    t = slot;
    u = slot < g.uslots ? (int)(slot * U / g.uslots) : 0;
    u1 = slot < g.uslots ? (int)((slot + 1) * U / g.uslots) : 0;
  }
  __device__ bool next(const TcArgs& g, Work& w) {
    if (t < g.full) {
      w = Work{t, 0, g.nch};
      t += g.slots;
      return true;
    }
    if (u >= u1) return false;
    w.tile = g.full + u / g.nch;
    w.c0 = u % g.nch;
    w.c1 = min(g.nch, w.c0 + (u1 - u));
    u += w.c1 - w.c0;
    return true;
  }
};

// x 2^e for -252 <= e <= 252, as two factors that are normal numbers
__device__ __forceinline__ float scale_pow2(float x, int e) {
  const int h = e >> 1;
  return x * __int_as_float((h + 127) << 23) * __int_as_float((e - h + 127) << 23);
}

constexpr int EPI_WARPS = 16, EPI0 = 2;
constexpr int P_THREADS = 32 * (EPI0 + EPI_WARPS);   // warp 0 TMA, 1 MMA, 2..17 epilogue
constexpr int EPI_GRP = EPI_WARPS / 4;               // warps that share a TMEM lane quarter
constexpr int EPI_B = BNMAX / 32 / EPI_GRP;          // 32-column blocks per warp
// How C is written. ROWS_BULK: n contiguous and 16-byte granules throughout; a warp stages 32 x 32
// blocks in shared memory and each lane sends its row by an asynchronous bulk copy (with plain
// stores the epilogue was as long as the MMAs of a K = 500 tile and did not overlap them).
// ROWS: n contiguous otherwise. LANES: a row per lane, for m contiguous (and any other) maps.
enum Out { ROWS_BULK = 0, ROWS = 1, LANES = 2 };
constexpr int EPI_LD = 36;                           // row stride (floats) of a warp's 32 x 32 block: 128-bit writes
constexpr int EPI_BLK = 32 * EPI_LD;                 // of a row per lane are conflict-free
constexpr int EPI_NBUF = 1;
constexpr int EPI_WARP = EPI_NBUF * EPI_BLK + 32 * EPI_B;   // floats per warp: blocks, and its columns' scales
constexpr int EPI_BYTES = EPI_WARPS * EPI_WARP * 4;
template <bool PAIR> __host__ __device__ constexpr int t_stages() { return PAIR ? 4 : 3; }
template <bool PAIR> __host__ __device__ constexpr int t_stage_bytes() { return TILE_A + (PAIR ? BNMAX / 2 : BNMAX) * ROWB; }
template <bool PAIR> __host__ __device__ constexpr int t_epi_off() { return t_stages<PAIR>() * t_stage_bytes<PAIR>(); }
template <bool PAIR> __host__ __device__ constexpr int t_smem_bytes() { return t_epi_off<PAIR>() + EPI_BYTES + 256 + 1024; }
static_assert(t_smem_bytes<false>() <= 227 * 1024 && t_smem_bytes<true>() <= 227 * 1024, "shared memory");

// Warp roles: one TMA thread per CTA, one MMA thread (cluster rank 0 issues for both CTAs of a
// pair; each CTA holds 128 rows of A and half of the tile's B rows), sixteen epilogue warps that
// keep the running sum of 128 rows x up to 256 columns in registers (64 per thread).
template <bool PAIR, int OUT>
__global__ void __launch_bounds__(P_THREADS, 1) k_gemm_f16x3(const __grid_constant__ CUtensorMap mapA,
                                                             const __grid_constant__ CUtensorMap mapB, TcArgs g) {
  constexpr int CS = PAIR ? 2 : 1;
  constexpr int ST = t_stages<PAIR>(), STB = t_stage_bytes<PAIR>();
  const uint32_t rank = PAIR ? cluster_rank() : 0;
  const bool issuer = rank == 0;
  // a CTA pair may not split up on a shared early exit, so only single CTAs return here
  if (!PAIR && *(volatile int*)g.err) return;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = (uint8_t*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* full = (uint64_t*)(smem + t_epi_off<PAIR>() + EPI_BYTES);
  uint64_t* empty = full + ST;
  uint64_t* accf = empty + ST;    // [2] chunk accumulated
  uint64_t* acce = accf + 2;      // [2] accumulator read
  uint64_t* drain = acce + 2;
  uint32_t* tmem_slot = (uint32_t*)(drain + 1);
  volatile int* abort_flag = (volatile int*)(tmem_slot + 1);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int slot = blockIdx.x / CS;
  const int bnh = g.bn / CS;      // B rows held by this CTA
  auto tile_mn = [&](int tile, int& m0, int& n0) {
    const int mt = g.m_fast ? tile % g.mt : tile / g.nt;
    const int nt = g.m_fast ? tile / g.mt : tile % g.nt;
    m0 = mt * (BM * CS) + (int)rank * BM;
    n0 = nt * g.bn;
  };

  if (threadIdx.x == 0) {
    for (int st = 0; st < ST; ++st) {
      mbar_init(&full[st], 1);
      mbar_init(&empty[st], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], EPI_WARPS * CS);
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    if constexpr (PAIR) {   // one warp of each CTA of the pair, collectively
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(2 * ACC_COLS));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    } else {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                   "r"(2 * ACC_COLS));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if constexpr (PAIR) cluster_sync_all();   // the peer's barriers are initialised before any remote arrival
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  int issued = 0;
  WorkIter wi(g, slot);
  Work w;
  if (warp == 0) {
    if (lane == 0) {
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&mapA) : "memory");
      asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&mapB) : "memory");
      bool ok = !g.hold;
      while (ok && wi.next(g, w)) {
        int m0, n0;
        tile_mn(w.tile, m0, n0);
        const int kb1 = min(w.c1 * CHB, g.nk);
        for (int kb = w.c0 * CHB; kb < kb1; ++kb, ++issued) {
          const int st = issued % ST;
          if (!mbar_wait(&empty[st], ((issued / ST) & 1) ^ 1, abort_flag)) { ok = false; break; }
          uint8_t* a = smem + st * STB;
          // the barrier of rank 0 counts the bytes of both CTAs (x: halves, a multiple of 128 bytes)
          if (issuer) mbar_arrive_expect_tx(&full[st], (uint32_t)(CS * (TILE_A + bnh * ROWB)));
          if constexpr (PAIR) {
            tma_load_2d_pair(a, &mapA, &full[st], kb * 2 * BK, m0);
            tma_load_2d_pair(a + TILE_A, &mapB, &full[st], kb * 2 * BK, n0 + (int)rank * bnh);
          } else {
            tma_load_2d(a, &mapA, &full[st], kb * 2 * BK, m0);
            tma_load_2d(a + TILE_A, &mapB, &full[st], kb * 2 * BK, n0);
          }
        }
      }
    }
  } else if (warp == 1) {
    if (issuer) {
      const bool leader = elect_one();   // 2 % faster than lane 0 by itself (3.68 -> 3.61 ms at 500 x 9936 x 108000)
      // D FP32; A, B FP16; N; M
      const uint32_t idesc = (1u << 4) | ((uint32_t)(g.bn >> 3) << 17) | ((uint32_t)((BM * CS) >> 4) << 24);
      constexpr uint16_t both = (1u << CS) - 1;
      int it = 0, lc = 0;
      bool ok = true;
      while (ok && wi.next(g, w)) {
        for (int c = w.c0; c < w.c1 && ok; ++c, ++lc) {
          const int buf = lc & 1;
          if (!mbar_wait_warp(&acce[buf], ((lc >> 1) & 1) ^ 1, abort_flag)) { ok = false; break; }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t d = tmem + (uint32_t)(buf * ACC_COLS);
          const int kb0 = c * CHB, kb1 = min(kb0 + CHB, g.nk);
          for (int kb = kb0; kb < kb1; ++kb, ++it) {
            const int st = it % ST;
            if (!mbar_wait_warp(&full[st], (it / ST) & 1, abort_flag)) { ok = false; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t a = sdesc(smem + st * STB), b = sdesc(smem + st * STB + TILE_A);
#pragma unroll
            for (int kk = 0; kk < BK / 16; ++kk) {   // hi at bytes 0..63 of a row, lo at 64..127
              const uint64_t h = 2 * kk, l = 4 + 2 * kk;
              if (leader) {
                mma_f16_ss<PAIR>(d, a + l, b + h, idesc, ((kb - kb0) | kk) ? 1u : 0u);
                mma_f16_ss<PAIR>(d, a + h, b + l, idesc, 1u);
                mma_f16_ss<PAIR>(d, a + h, b + h, idesc, 1u);
              }
            }
            if (leader) mma_commit<PAIR>(&empty[st], both);
          }
          if (ok && leader) mma_commit<PAIR>(&accf[buf], both);
        }
      }
      if (leader) mma_commit<PAIR>(drain, 1);
      const unsigned long long t0 = clock64();
      while (!mbar_try_wait(drain, 0) && clock64() - t0 < WAIT_LIMIT) {
      }
    }
    __syncwarp();
  } else {
    // epilogue: TMEM lane quarter = warp % 4; the 32-column blocks h, h + EPI_GRP, ...
    const int q = warp % 4, h = (warp - EPI0) / 4;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const int nblk = g.bn / 32;
    float* blk = (float*)(smem + t_epi_off<PAIR>()) + (warp - EPI0) * EPI_WARP;
    float* scol = blk + EPI_NBUF * EPI_BLK;   // 2^-e of this warp's columns in the current chunk
    int bulk = 0;                             // bulk copies in flight use the blocks in turn
    int lc = 0;
    bool ok = true;
    while (ok && wi.next(g, w)) {
      int m0, n0;
      tile_mn(w.tile, m0, n0);
      const int m = m0 + q * 32 + lane;
      const bool mrow = m < g.M;
      float run[EPI_B][32];
#pragma unroll
      for (int i = 0; i < EPI_B; ++i)
#pragma unroll
        for (int j = 0; j < 32; ++j) run[i][j] = 0.f;
      for (int c = w.c0; c < w.c1; ++c, ++lc) {
        const int buf = lc & 1;
        const float sa = mrow ? __ldg(g.inva + c * g.sca + m) : 1.f;
        // the product of two scales is a normal number unless an operand is near the ends of FP32
        bool mild = abs((int)(__float_as_uint(sa) >> 23) - 127) <= 60;
        __syncwarp();
#pragma unroll
        for (int i = 0; i < EPI_B; ++i)
          if (h + EPI_GRP * i < nblk) {
            const int n = n0 + (h + EPI_GRP * i) * 32 + lane;
            const float sb = n < g.N ? __ldg(g.invb + c * g.scb + n) : 1.f;
            mild = mild && abs((int)(__float_as_uint(sb) >> 23) - 127) <= 60;
            scol[i * 32 + lane] = sb;
          }
        mild = __all_sync(0xffffffffu, mild);
        __syncwarp();   // the lanes' scales are written: every lane reads all of them
        if (!__all_sync(0xffffffffu, mbar_wait_sleep(&accf[buf], (lc >> 1) & 1, abort_flag))) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int i = 0; i < EPI_B; ++i)
          if (h + EPI_GRP * i < nblk) {
#pragma unroll
            for (int t = 0; t < 32; t += 16) {   // 16 columns at a time
              uint32_t r[16];
              tmem_ld16(tmem + lane_base + (uint32_t)(buf * ACC_COLS + (h + EPI_GRP * i) * 32 + t), r);
              tmem_wait_tie(r);
              if (mild) {
#pragma unroll
                for (int j = 0; j < 16; j += 4) {
                  const float4 s = *(const float4*)(scol + i * 32 + t + j);
                  run[i][t + j] = fmaf(__uint_as_float(r[j]), s.x * sa, run[i][t + j]);
                  run[i][t + j + 1] = fmaf(__uint_as_float(r[j + 1]), s.y * sa, run[i][t + j + 1]);
                  run[i][t + j + 2] = fmaf(__uint_as_float(r[j + 2]), s.z * sa, run[i][t + j + 2]);
                  run[i][t + j + 3] = fmaf(__uint_as_float(r[j + 3]), s.w * sa, run[i][t + j + 3]);
                }
              } else {   // the two powers of two applied as one exponent
                const int ea = (int)(__float_as_uint(sa) >> 23) - 127;
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                  const int eb = (int)(__float_as_uint(scol[i * 32 + t + j]) >> 23) - 127;
                  run[i][t + j] += scale_pow2(__uint_as_float(r[j]), ea + eb);
                }
              }
            }
          }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive_issuer<PAIR>(&acce[buf], rank);
      }
      if (!ok || __shfl_sync(0xffffffffu, *abort_flag, 0)) break;   // warp-uniform
      if (w.c1 - w.c0 < g.nch) {   // a piece of a cut tile: rows fastest, added up by k_join_pieces
        float* p = g.part + (int64_t)(2 * slot + (w.c0 > 0 ? 0 : 1)) * (g.bn * BM * CS) + rank * BM + q * 32 + lane;
#pragma unroll
        for (int i = 0; i < EPI_B; ++i)
          if (h + EPI_GRP * i < nblk)
#pragma unroll
            for (int j = 0; j < 32; ++j) p[(int64_t)((h + EPI_GRP * i) * 32 + j) * (BM * CS)] = run[i][j];
        continue;
      }
      float* row = g.C + (mrow ? (int64_t)(m / g.mdiv) * g.c0 + (int64_t)(m % g.mdiv) * g.c1 : 0);
#pragma unroll
      for (int i = 0; i < EPI_B; ++i) {
        const int nb0 = n0 + (h + EPI_GRP * i) * 32;
        if (h + EPI_GRP * i < nblk && nb0 < g.N) {
          int nr = nb0 % g.ndiv;
          float* dst = row + (int64_t)(nb0 / g.ndiv) * g.c2 + (int64_t)nr * g.c3;
          if constexpr (OUT == LANES) {
            if (mrow) {
#pragma unroll
              for (int j = 0; j < 32; ++j) {
                if (nb0 + j < g.N) {
                  if (g.accumulate) atomicAdd(dst, run[i][j]);
                  else *dst = run[i][j];
                }
                dst += g.c3;
                if (++nr == g.ndiv) {
                  nr = 0;
                  dst += g.c2 - (int64_t)g.ndiv * g.c3;
                }
              }
            }
          } else {
            float* sb = blk + (OUT == ROWS_BULK ? (bulk++ % EPI_NBUF) * EPI_BLK : 0);
            if constexpr (OUT == ROWS_BULK) bulk_wait_read<EPI_NBUF - 1>();   // this block's previous copy has read it
            __syncwarp();
#pragma unroll
            for (int j = 0; j < 32; j += 4)
              *(float4*)(sb + lane * EPI_LD + j) = make_float4(run[i][j], run[i][j + 1], run[i][j + 2], run[i][j + 3]);
            if constexpr (OUT == ROWS_BULK) {
              asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
              // this lane's row: a run of ndiv may end inside it (runs are at least 32 long)
              const int left = min(32, g.N - nb0), n1 = min(left, g.ndiv - nr);
              const float* src = sb + lane * EPI_LD;
              if (mrow) {
                bulk_s2g(dst, src, 4 * n1, g.accumulate);
                if (n1 < left) bulk_s2g(dst + n1 + g.c2 - g.ndiv, src + n1, 4 * (left - n1), g.accumulate);
              }
              bulk_commit();
            } else {
              __syncwarp();
              const int n = nb0 + lane;
              const bool ncol = n < g.N;
              const int64_t no = ncol ? (int64_t)(n / g.ndiv) * g.c2 + n % g.ndiv : 0;
              const int mleft = min(32, g.M - (m0 + q * 32));
#pragma unroll 4
              for (int r = 0; r < 32; ++r) {
                float* d = (float*)__shfl_sync(0xffffffffu, (unsigned long long)row, r) + no;
                if (r < mleft && ncol) {
                  if (g.accumulate) atomicAdd(d, sb[r * EPI_LD + lane]);
                  else *d = sb[r * EPI_LD + lane];
                }
              }
            }
          }
        }
      }
    }
    if constexpr (OUT == ROWS_BULK) bulk_wait_all();   // the copies read this CTA's shared memory
  }

  // every role has left its loop (finished or aborted) once all threads meet here; only then is
  // the abort flag final
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*abort_flag) {
    if (warp == 0 && lane == 0 && issuer) {   // wait (bounded) for the TMA loads still in flight
      for (int it = issued > ST ? issued - ST : 0; it < issued; ++it) {
        const unsigned long long t0 = clock64();
        while (!mbar_try_wait(&full[it % ST], (it / ST) & 1) && clock64() - t0 < WAIT_LIMIT) {
        }
      }
    }
    if (threadIdx.x == 0) atomicExch(g.err, 1);
  }
  __syncthreads();
  // the pair's MMAs read this CTA's shared memory and write its TMEM, the peer's loads count on
  // this CTA's barriers: neither CTA frees or exits before both are here
  if constexpr (PAIR) cluster_sync_all();
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if constexpr (PAIR)
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * ACC_COLS));
    else
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * ACC_COLS));
  }
}

// The pieces of the tiles cut between slots, added without rounding error in slot order and written through the
// output map. blockIdx.x = b - 1 for the cut between slots b - 1 and b; the first cut inside a tile
// stands for the tile. Blocks of 32 x 32 outputs go through shared memory, so that reads run
// along m and stores along the contiguous index of C.
__global__ void __launch_bounds__(256) k_join_pieces(TcArgs g, int rows) {
  __shared__ float t[32][33];
  const int64_t U = (int64_t)(g.ntiles - g.full) * g.nch;
  const int64_t b = blockIdx.x + 1, cut = b * U / g.uslots;
  if (cut % g.nch == 0) return;
  const int64_t tile = cut / g.nch, first = tile * g.nch, last = first + g.nch - 1;
  if ((b - 1) * U / g.uslots > first) return;       // an earlier cut of this tile stands for it
  const int64_t s0 = b - 1;                         // the slots that hold its pieces: s0 .. s0 + np - 1
  const int np = (int)(((last + 1) * g.uslots - 1) / U - s0) + 1;
  const int64_t ti = g.full + tile;
  const int64_t mt = g.m_fast ? ti % g.mt : ti / g.nt, nt = g.m_fast ? ti / g.mt : ti % g.nt;
  const int64_t m0 = mt * rows, n0 = nt * (int64_t)g.bn, psz = (int64_t)g.bn * rows;
  const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;
  for (int blk = blockIdx.y; blk < (rows / 32) * (g.bn / 32); blk += gridDim.y) {
    const int r0 = blk % (rows / 32) * 32, c0 = blk / (rows / 32) * 32;
    if (m0 + r0 >= g.M || n0 + c0 >= g.N) continue;
    __syncthreads();
    const float* p = g.part + (2 * s0 + 1) * psz + (int64_t)(c0 + ty) * rows + r0 + tx;   // the tile's head
    float hi[4], lo[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      hi[c] = p[(int64_t)(8 * c) * rows];
      lo[c] = 0.f;
    }
    p += psz;                                                                             // slot s0 + 1, its tail
#pragma unroll 8
    for (int s = 1; s < np; ++s, p += 2 * psz)
#pragma unroll
      for (int c = 0; c < 4; ++c) {   // error-free sum (Knuth's two-sum): FP64 adds cost ten times as much here
        const float x = p[(int64_t)(8 * c) * rows], z = hi[c] + x, v = z - hi[c];
        lo[c] += (hi[c] - (z - v)) + (x - v);
        hi[c] = z;
      }
#pragma unroll
    for (int c = 0; c < 4; ++c) t[ty + 8 * c][tx] = hi[c] + lo[c];
    __syncthreads();
    for (int i = ty; i < 32; i += 8) {
      const int c = g.c3 == 1 ? tx : i, r = g.c3 == 1 ? i : tx;
      const int64_t m = m0 + r0 + r, n = n0 + c0 + c;
      if (m >= g.M || n >= g.N) continue;
      const int mi = (int)m, ni = (int)n;
      float* dst = g.C + (int64_t)(mi / g.mdiv) * g.c0 + (int64_t)(mi % g.mdiv) * g.c1 + (int64_t)(ni / g.ndiv) * g.c2 + (int64_t)(ni % g.ndiv) * g.c3;
      *dst = g.accumulate ? *dst + t[c][r] : t[c][r];
    }
  }
}

// ---------------------------------------------------------------- host side
using EncodeTiled = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                 const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiled encoder() {
  static EncodeTiled fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiled)p;
  });
  FP_CHECK(fn != nullptr, FPEPS_ERR_CUDA, "cuTensorMapEncodeTiled unavailable");
  return fn;
}

// map of a split operand: rows of nk k-blocks of 64 halves; rows outside the matrix read as zeros
CUtensorMap make_map(const __half* base, int64_t rows, int64_t nk, int box_rows) {
  CUtensorMap m;
  cuuint64_t dims[2] = {(cuuint64_t)(nk * 2 * BK), (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)nk * ROWB};
  cuuint32_t box[2] = {(cuuint32_t)(2 * BK), (cuuint32_t)box_rows};
  cuuint32_t es[2] = {1, 1};
  CUresult r = encoder()(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, (void*)base, dims, strides, box, es,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  FP_CHECK(r == CUDA_SUCCESS, FPEPS_ERR_CUDA, "cuTensorMapEncodeTiled failed");
  return m;
}

// SMs, and CTA pairs the GPU holds at once (clusters of two CTAs, one CTA per SM; 0 if the pair kernel
// cannot be launched). Asking for them also prepares the kernels for launches in this context.
struct Limits {
  int sms, pairs;
};
template <bool PAIR>
void allow_smem() {
  FP_CUDA(cudaFuncSetAttribute(k_gemm_f16x3<PAIR, ROWS_BULK>, cudaFuncAttributeMaxDynamicSharedMemorySize, t_smem_bytes<PAIR>()));
  FP_CUDA(cudaFuncSetAttribute(k_gemm_f16x3<PAIR, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, t_smem_bytes<PAIR>()));
  FP_CUDA(cudaFuncSetAttribute(k_gemm_f16x3<PAIR, LANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, t_smem_bytes<PAIR>()));
}
Limits limits() {
  static PerContext<Limits> per;
  return per.get([] {
    allow_smem<false>();
    allow_smem<true>();
    int dev = 0;
    Limits l{0, 0};
    FP_CUDA(cudaGetDevice(&dev));
    FP_CUDA(cudaDeviceGetAttribute(&l.sms, cudaDevAttrMultiProcessorCount, dev));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(l.sms & ~1));
    cfg.blockDim = dim3(P_THREADS);
    cfg.dynamicSmemBytes = t_smem_bytes<true>();
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&l.pairs, k_gemm_f16x3<true, LANES>, &cfg) != cudaSuccess) {
      (void)cudaGetLastError();
      l.pairs = 0;
    }
    return l;
  });
}

// Tile shape and schedule of one product: the estimated cycles of the busiest slot. A k-block costs
// six MMAs of BN / 2 cycles (at least 64), a tile its epilogue, a cut last wave the second kernel.
struct Plan {
  bool pair = false;
  int bn = BNMAX;
  int64_t mt = 0, nt = 0, slots = 0, full = 0, nk = 0, nch = 0;
};
Plan plan_of(int64_t M, int64_t N, int64_t K) {
  Plan best;
  double cost = 1e300;
  const int64_t nk = (K + BK - 1) / BK, nch = (nk + CHB - 1) / CHB;
  const Limits lim = limits();
  for (int pr = 0; pr < 2; ++pr) {
    if (pr && (M <= BM || lim.pairs <= 0)) continue;
    const int64_t most = pr ? lim.pairs : lim.sms;
    const int64_t mt = (M + BM * (1 + pr) - 1) / (BM * (1 + pr));
    for (int cap = BNMAX; cap >= 32; cap /= 2) {
      const int64_t w = (N + cap - 1) / cap;
      const int bn = (int)(((N + w - 1) / w + 31) / 32 * 32);
      const int64_t nt = (N + bn - 1) / bn, tiles = mt * nt;
      // single CTAs read all of B from their own shared memory: ~1.3 times the pair's cycles
      const double kb = 6.0 * std::max(64.0, bn / 2.0) * (pr ? 1.0 : 1.3), tail = 1500.0 + 12.0 * bn;
      for (int cut = 0; cut < 2; ++cut) {
        const int64_t full = cut ? tiles / most * most : tiles;
        const int64_t units = (tiles - full) * nch;
        if (cut && (units == 0 || nch == 1)) continue;
        const int64_t slots = cut && full == 0 ? std::min(most, units) : std::min(most, cut ? most : tiles);
        double c = (double)((full + slots - 1) / slots) * (nk * kb + tail);
        if (cut) c += (double)((units + slots - 1) / slots) * CHB * kb + 2 * tail + 9000.0;
        if (c < 0.97 * cost) {
          cost = c;
          best.pair = pr != 0;
          best.bn = bn;
          best.mt = mt;
          best.nt = nt;
          best.slots = slots;
          best.full = full;
          best.nk = nk;
          best.nch = nch;
        }
      }
    }
  }
  return best;
}

template <bool PAIR, int OUT>
void launch_gemm(cudaStream_t s, int64_t slots, const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& g) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(slots * (PAIR ? 2 : 1)));
  cfg.blockDim = dim3(P_THREADS);
  cfg.dynamicSmemBytes = t_smem_bytes<PAIR>();
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = PAIR ? 1 : 0;
  FP_CUDA(cudaLaunchKernelEx(&cfg, k_gemm_f16x3<PAIR, OUT>, ma, mb, g));
}

size_t up256(size_t b) { return (b + 255) / 256 * 256; }

// Whether a product runs on planes (this file) or splits on chip (gemm_onchip.cu), both estimated
// in microseconds. Planes: one pass over both operands (8 bytes per element at ~6.5 TB/s), then
// ~500 TFLOP/s, and two or three launches. On chip: ~240 TFLOP/s, one launch. Measured on GB300,
// on chip / planes: 108000 x 9936 x 500 4.32 / 2.38 ms, 500 x 9936 x 108000 4.41 / 3.66 ms,
// 8192^3 4.06 / 2.19 ms, but 256 x 38304 x 36864 2.80 / 3.34 ms (the large operand is used by one
// row of tiles) and 100 x 5000 x 3000 88 / 121 us.
bool on_planes(int64_t M, int64_t N, int64_t K) {
  const double f = 2.0 * (double)M * (double)N * (double)K;
  return 8.0 * (double)(M + N) * (double)K / 6.5e6 + f / 500e6 + 20.0 < f / 240e6;
}

// A long sum runs in panels of K, whose split operands stay within about half a gigabyte.
int64_t panel_of(int64_t M, int64_t N, int64_t K) {
  const int64_t fit = std::max<int64_t>(2048, ((512LL << 20) / (4 * (M + N))) / 2048 * 2048);
  const int64_t np = (K + fit - 1) / fit;
  return ((K + np - 1) / np + SEG - 1) / SEG * SEG;   // whole scale segments
}

// scratch: header, pieces of cut tiles, then the split operands and their scales; the on-chip split of
// graded operands uses the same bytes after them
size_t part_bytes(const Plan& p) {
  return p.full < p.mt * p.nt ? up256((size_t)2 * p.slots * p.bn * BM * (p.pair ? 2 : 1) * 4) : 0;
}
size_t split_bytes(int64_t rows, int64_t K) {
  const int64_t nk = (K + BK - 1) / BK, nch = (nk + CHB - 1) / CHB;
  return up256((size_t)rows * nk * ROWB) + up256((size_t)rows * nch * 4);
}

Grading* grading_of(void* scratch) { return (Grading*)((int*)scratch + 4); }

void run_planes(cudaStream_t s, int64_t M, int64_t N, int64_t K, const SplitMat& A, const SplitMat& B, float* C, OutMap om,
                void* scratch, bool accumulate, bool hold) {
  const Plan p = plan_of(M, N, K);
  const int64_t tiles = p.mt * p.nt;
  FP_CHECK(tiles < (1LL << 30), FPEPS_ERR_UNSUPPORTED, "tensor-core GEMM: grid too large");
  FP_CHECK(om.mdiv > 0 && om.ndiv > 0, FPEPS_ERR_ARG, "tensor-core GEMM: bad output map");
  const int cs = p.pair ? 2 : 1;
  const CUtensorMap ma = make_map((const __half*)A.planes, M, p.nk, BM), mb = make_map((const __half*)B.planes, N, p.nk, p.bn / cs);
  TcArgs g;
  g.M = (int)M; g.N = (int)N; g.C = C; g.err = (int*)scratch;
  g.mdiv = (int)std::min<int64_t>(om.mdiv, INT32_MAX);   // m, n < 2^31 - 1: a larger divisor never divides
  g.ndiv = (int)std::min<int64_t>(om.ndiv, INT32_MAX);
  g.c0 = om.c0; g.c1 = om.c1; g.c2 = om.c2; g.c3 = om.c3;
  const bool granules = om.ndiv % 4 == 0 && om.ndiv >= 32 && N % 4 == 0 && om.c0 % 4 == 0 && om.c1 % 4 == 0 &&
                        om.c2 % 4 == 0 && ((uintptr_t)C % 16) == 0;
  const int out = om.c3 != 1 ? LANES : granules ? ROWS_BULK : ROWS;
  g.inva = A.inv; g.invb = B.inv;
  g.sca = A.inv_stride; g.scb = B.inv_stride;
  g.part = (float*)((char*)scratch + kTcHeader);
  g.bn = p.bn;
  g.mt = (int)p.mt; g.nt = (int)p.nt;
  g.m_fast = g.mt <= g.nt ? 1 : 0;
  g.full = (int)p.full; g.ntiles = (int)tiles; g.slots = (int)p.slots;
  g.uslots = (int)std::max<int64_t>(1, std::min(p.slots, (tiles - p.full) * p.nch));   // every one gets a unit
  g.nk = (int)p.nk; g.nch = (int)p.nch;
  g.accumulate = accumulate ? 1 : 0;
  g.hold = hold ? 1 : 0;
  if (p.pair) (out == LANES ? launch_gemm<true, LANES> : out == ROWS ? launch_gemm<true, ROWS> : launch_gemm<true, ROWS_BULK>)(s, p.slots, ma, mb, g);
  else (out == LANES ? launch_gemm<false, LANES> : out == ROWS ? launch_gemm<false, ROWS> : launch_gemm<false, ROWS_BULK>)(s, p.slots, ma, mb, g);
  FP_LAUNCH();
  if (g.full < tiles && g.uslots > 1) {
    k_join_pieces<<<dim3((unsigned)(g.uslots - 1), 64), 256, 0, s>>>(g, BM * cs);
    FP_LAUNCH();
  }
}

}  // namespace

bool gemm_tc_supported(int64_t M, int64_t N, int64_t K, int64_t lda, int64_t ldb) {
  // rows on 16-byte boundaries (128-bit loads of the splitting pass), at least one full k-block
  return M >= 1 && N >= 1 && K >= BK && (lda % 4) == 0 && (ldb % 4) == 0 && lda >= K && ldb >= K &&
         M < (1LL << 31) - 1024 && N < (1LL << 31) - 1024 && K < (1LL << 31);
}

size_t gemm_tc_scratch_bytes(int64_t M, int64_t N, int64_t K) {
  if (!on_planes(M, N, K)) return gemm_onchip_scratch_bytes(M, N, K);
  const int64_t kp = panel_of(M, N, K), last = K - (K - 1) / kp * kp;
  return std::max(gemm_onchip_scratch_bytes(M, N, K),
                  kTcHeader + std::max(part_bytes(plan_of(M, N, std::min(kp, K))), part_bytes(plan_of(M, N, last))) +
                      split_bytes(M, std::min(kp, K)) + split_bytes(N, std::min(kp, K)));
}

void gemm_tc(cudaStream_t s, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
             int64_t ldb, float* C, OutMap om, void* scratch, size_t scratch_bytes, int mark, bool settle) {
  FP_CHECK(((uintptr_t)A % 16) == 0 && ((uintptr_t)B % 16) == 0, FPEPS_ERR_ARG, "tensor-core GEMM: operand alignment");
  ProfToken pt = prof_begin(PROF_GEMM_TC, s, 2.0 * M * N * K, 4.0 * ((double)M * K + (double)N * K + (double)M * N));
  if (!on_planes(M, N, K) || scratch_bytes < gemm_tc_scratch_bytes(M, N, K)) {
    gemm_onchip(s, M, N, K, A, lda, B, ldb, C, om, scratch, scratch_bytes);
    prof_end(pt, s);
    return;
  }
  const int64_t kp = panel_of(M, N, K);
  for (int64_t k0 = 0; k0 < K; k0 += kp) {
    const int64_t k = std::min(kp, K - k0), nk = (k + BK - 1) / BK, nch = (nk + CHB - 1) / CHB;
    char* base = (char*)scratch + kTcHeader + part_bytes(plan_of(M, N, k));
    SplitOp oa{A + k0, M, lda, (__half*)base, (float*)(base + up256((size_t)M * nk * ROWB))};
    base += split_bytes(M, k);
    SplitOp ob{B + k0, N, ldb, (__half*)base, (float*)(base + up256((size_t)N * nk * ROWB))};
    k_split_planes<<<(unsigned)std::min<int64_t>(((M + N) * nch + 7) / 8, 152 * 32), 256, 0, s>>>(oa, ob, k, (unsigned)nk, (unsigned)nch,
                                                                                                         grading_of(scratch), mark);
    FP_LAUNCH();
    run_planes(s, M, N, k, SplitMat{oa.planes, oa.inv, M}, SplitMat{ob.planes, ob.inv, N}, C, om, scratch, k0 > 0, false);
  }
  if (settle) gemm_tc_settle(s, M, N, K, A, lda, B, ldb, C, om, scratch, scratch_bytes, mark);
  prof_end(pt, s);
}

void gemm_tc_settle(cudaStream_t s, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
                    int64_t ldb, float* C, OutMap om, void* scratch, size_t scratch_bytes, int mark) {
  if (!on_planes(M, N, K) || scratch_bytes < gemm_tc_scratch_bytes(M, N, K)) return;
  const SplitOp oa{A, M, lda, nullptr, nullptr}, ob{B, N, ldb, nullptr, nullptr};
  k_uneven<<<152, 256, 0, s>>>(oa, ob, K, (unsigned)((K + SEG - 1) / SEG), grading_of(scratch), mark);
  FP_LAUNCH();
  gemm_onchip(s, M, N, K, A, lda, B, ldb, C, om, scratch, scratch_bytes, false, grading_of(scratch), mark);
}

void gemm_tc_hold(cudaStream_t s, int64_t M, int64_t N, int64_t K, void* planes, float* C, void* scratch) {
  const SplitMat z{planes, (const float*)planes, 0};
  run_planes(s, M, N, K, z, z, C, out_rowmajor(M, N, N), scratch, false, true);
}

}  // namespace fpeps
