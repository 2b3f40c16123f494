// SVD of the small dense matrices (FP64): one-sided Jacobi.
//
// Hestenes' method with the cyclic round-robin ordering; each rotation makes two columns
// orthogonal (Demmel and Veselic 1992). The path always applies it to the transposed triangular
// factor of a QR (the preconditioned form of Drmac and Veselic 2008).
//
// FP64 is the limit: this part does two FP64 FMAs per cycle and SM against 128 in FP32, and nine
// to eleven FP64 sweeps at k = 510 cost 56 ms. Sweeps in FP64 are only needed at the end, so
// matrices of more than kDirect columns go through
//   1. Jacobi in FP32 on a copy of M (k_jacobi32, k_jacobi32_blk), the rotations accumulated in
//      double-float (two FP32 numbers, ~47 bits): V0. Every rotation acts on two columns at their
//      own scale, so graded matrices lose nothing (a mixed-precision Jacobi preconditioner; Gao,
//      Ma and Shao 2022).
//   2. V = V0 (3/2 - V0^T V0 / 2) in FP64, one Newton-Schulz step: orthonormal to FP64 rounding;
//      M <- M V, M at unit scale from here on (a power of two, put back on the singular values).
//   3. G = M^T M gives every remaining angle at once: S_pq = t(G_pp, G_qq, G_pq), the Jacobi
//      tangents as a skew matrix, and M, V <- M, V exp(S) by matrix products (the first-order
//      correction of Ogita and Aishima 2020, with the exponential to fourth order so that V stays
//      orthonormal). The largest |cos| falls quadratically: ~1e-6, ~1e-9, then below what the FP64
//      method itself stops at. At most three such steps.
//   4. If a pair's angle is not small (close singular values) or |cos| has not fallen, the FP64
//      Jacobi sweeps finish the job from there; the same convergence test decides in both.
// Steps 2 and 3 are FP64 matrix products, spread over the whole GPU.
#include <cooperative_groups.h>

#include <algorithm>

#include "common.cuh"

namespace fpeps {
namespace {

// One round of the one-sided Jacobi method on the columns of M (col-major,
// k x k) with the accumulated right rotations in V. Pairs of the round-robin
// schedule: player positions 0..kk-1 (kk even), position 0 fixed.
__device__ __forceinline__ int rr_player(int pos, int round, int kk) {
  if (pos == 0) return 0;
  return 1 + ((pos - 1 + round) % (kk - 1));
}

__global__ void __launch_bounds__(1024) k_jacobi_svd(double* M, double* V, int k, int max_sweeps, double eps,
                                                      const int* skip, bool init) {
  if (skip && *skip) return;
  const int kk = (k % 2) ? k + 1 : k;   // dummy column k when odd
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nwarp = blockDim.x / 32;
  __shared__ int rotated;
  __shared__ double fro2;
  if (init)
    for (int e = threadIdx.x; e < k * k; e += blockDim.x) V[e] = ((e / k) == (e % k)) ? 1.0 : 0.0;
  if (threadIdx.x == 0) {
    double f = 0;
    for (int64_t e = 0; e < (int64_t)k * k; ++e) f = fma(M[e], M[e], f);
    fro2 = f;
  }
  __syncthreads();
  // a column whose squared norm is below 1e-30 of the whole matrix carries no
  // resolvable direction: rotations against it only stir rounding noise
  const double tiny = 1e-30 * fro2;
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    if (threadIdx.x == 0) rotated = 0;
    __syncthreads();
    for (int round = 0; round < kk - 1; ++round) {
      for (int pr = warp; pr < kk / 2; pr += nwarp) {
        int a = rr_player(pr, round, kk), b = rr_player(kk - 1 - pr, round, kk);
        int p = min(a, b), q = max(a, b);
        if (q >= k) continue;
        double* mp = M + (int64_t)p * k;
        double* mq = M + (int64_t)q * k;
        double al = 0, be = 0, ga = 0;
        for (int i = lane; i < k; i += 32) {
          double x = mp[i], y = mq[i];
          al = fma(x, x, al); be = fma(y, y, be); ga = fma(x, y, ga);
        }
        for (int o = 16; o; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          ga += __shfl_xor_sync(0xffffffffu, ga, o);
        }
        if (ga == 0.0 || fmin(al, be) <= tiny || fabs(ga) <= eps * sqrt(al) * sqrt(be)) continue;
        double zeta = (be - al) / (2.0 * ga);
        double t = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
        double c = 1.0 / sqrt(1.0 + t * t), s = c * t;
        for (int i = lane; i < k; i += 32) {
          double x = mp[i], y = mq[i];
          mp[i] = c * x - s * y;
          mq[i] = s * x + c * y;
          double vx = V[(int64_t)p * k + i], vy = V[(int64_t)q * k + i];
          V[(int64_t)p * k + i] = c * vx - s * vy;
          V[(int64_t)q * k + i] = s * vx + c * vy;
        }
        if (lane == 0) rotated = 1;
      }
      __syncthreads();
    }
    if (!rotated) break;
    __syncthreads();
  }
  // reaching the sweep cap leaves the columns orthogonal to rounding level; it is not an error
}

// The same method spread over the whole GPU, in blocks of two columns (block b:
// columns 2b and 2b + 1). A round-robin schedule over the blocks gives every CTA a
// pair of blocks (A, B) per round; the CTA copies their four columns of M and of V to
// shared memory and rotates the four cross pairs, two at a time ((a0,b0) (a1,b1), then
// (a0,b1) (a1,b0)), after first rotating each block's own pair in the first round of a
// sweep. Every column pair is visited once per sweep, as in the scalar cyclic order,
// with one grid barrier per round of blocks. Each rotation is carried by two warps (one
// half of the rows each, partial dot products exchanged in shared memory), so the four
// warps of a CTA keep all four FP64 pipes of the SM busy: FP64 is the limit here (~2 FMA
// per cycle per SM on this part; a rotation of two length-k columns of M and of V costs
// ~11 k FMA).
// ws[0..1]: sweep rotation counters (two, alternating), ws[2]: squared Frobenius norm,
// ws[3]: sweeps used, ws[4..5]: counters of rotations above sqrt(big2) (alternating).
constexpr int JB_THREADS = 128;

// rotation of local columns (p, q) by the two warps h = 0, 1 of a pair slot: rows
// [h * half, (h + 1) * half); part[6] holds the two halves' (alpha, beta, gamma)
// *big (if given) is set when the rotation's |gamma| / sqrt(alpha beta) exceeds sqrt(big2)
__device__ __forceinline__ bool jacobi_rotate_split(double* __restrict__ mp, double* __restrict__ mq,
                                                    double* __restrict__ vp, double* __restrict__ vq, int k, int h,
                                                    int lane, double* part, double eps, double tiny, bool* big,
                                                    double big2) {
  const int half = (k + 1) / 2, i0 = h * half, i1 = min(k, i0 + half);
  double al = 0, be = 0, ga = 0;
  for (int i = i0 + lane; i < i1; i += 32) {
    const double x = mp[i], y = mq[i];
    al = fma(x, x, al);
    be = fma(y, y, be);
    ga = fma(x, y, ga);
  }
  for (int o = 16; o; o >>= 1) {
    al += __shfl_xor_sync(0xffffffffu, al, o);
    be += __shfl_xor_sync(0xffffffffu, be, o);
    ga += __shfl_xor_sync(0xffffffffu, ga, o);
  }
  if (lane == 0) {
    part[3 * h + 0] = al;
    part[3 * h + 1] = be;
    part[3 * h + 2] = ga;
  }
  __syncthreads();
  // both warps add the halves in the same order, so they take the same decision and angle
  al = part[0] + part[3];
  be = part[1] + part[4];
  ga = part[2] + part[5];
  // |gamma| <= eps sqrt(alpha beta) tested squared: FP64 sqrt and division are long serial
  // latencies here (~680 and ~430 cycles), so the angle takes one of each plus one rsqrt:
  // tan = sign(d) 2 gamma / (|d| + sqrt(d^2 + 4 gamma^2)), d = beta - alpha, which is
  // sign(zeta) / (|zeta| + sqrt(1 + zeta^2)) with zeta = d / (2 gamma)
  const bool rot = !(ga == 0.0 || fmin(al, be) <= tiny || ga * ga <= eps * eps * al * be);
  if (rot) {
    if (big && ga * ga > big2 * al * be) *big = true;
    const double d = be - al, g2 = 2.0 * ga;
    const double t = (d >= 0 ? g2 : -g2) / (fabs(d) + sqrt(fma(d, d, g2 * g2)));
    const double c = rsqrt(fma(t, t, 1.0)), sn = c * t;
    for (int i = i0 + lane; i < i1; i += 32) {
      const double x = mp[i], y = mq[i], a = vp[i], b = vq[i];
      mp[i] = c * x - sn * y;
      mq[i] = sn * x + c * y;
      vp[i] = c * a - sn * b;
      vq[i] = sn * a + c * b;
    }
  }
  return rot;
}

__global__ void __launch_bounds__(JB_THREADS) k_jacobi_svd_blk(double* M, double* V, int k, int max_sweeps,
                                                                double eps, double big2, const int* skip, bool init,
                                                                unsigned long long* ws) {
  if (skip && *skip) return;   // the same for every block: no barrier is entered
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  extern __shared__ double jsh[];   // M columns [4][k], V columns [4][k], partial dots [2][6]
  double* sm = jsh;
  double* sv = jsh + 4 * (int64_t)k;
  double* part = jsh + 8 * (int64_t)k;
  const int nb = (k + 1) / 2, nbe = nb + (nb & 1);   // blocks; a dummy block when nb is odd
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int slot = warp / 2, h = warp % 2;           // pair slot and row half of this warp
  double* fro2p = (double*)&ws[2];
  if (init)
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)k * k; e += (int64_t)gridDim.x * blockDim.x)
      V[e] = ((e / k) == (e % k)) ? 1.0 : 0.0;
  if (blockIdx.x == 0) {   // ||M||_F^2 by block 0
    __shared__ double red[JB_THREADS / 32];
    double f = 0;
    for (int64_t e = threadIdx.x; e < (int64_t)k * k; e += blockDim.x) f = fma(M[e], M[e], f);
    for (int o = 16; o; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (lane == 0) red[warp] = f;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0;
      for (int w = 0; w < JB_THREADS / 32; ++w) t += red[w];
      *fro2p = t;
      ws[0] = ws[1] = ws[4] = ws[5] = 0;
    }
  }
  grid.sync();
  const double tiny = 1e-30 * (*fro2p);
  // The rotation counter of sweep s lives in ws[s & 1] (its count of rotations above
  // sqrt(big2) in ws[4 + (s & 1)]); every block reads it after the last
  // round and a further barrier follows, so all blocks take the same break decision; the slot
  // is cleared for sweep s+2 at round 1 of sweep s+1, after those reads.
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    for (int round = 0; round < nbe - 1; ++round) {
      if (round == 1 && blockIdx.x == 0 && threadIdx.x == 0) ws[(sweep + 1) & 1] = ws[4 + ((sweep + 1) & 1)] = 0;
      const int A = rr_player((int)blockIdx.x, round, nbe), B = rr_player(nbe - 1 - (int)blockIdx.x, round, nbe);
      // local columns 0, 1 (block A) and 2, 3 (block B); -1: absent
      int col[4];
      col[0] = 2 * A;
      col[1] = 2 * A + 1;
      col[2] = 2 * B;
      col[3] = 2 * B + 1;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (col[j] >= k) col[j] = -1;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        for (int i = threadIdx.x; i < k; i += blockDim.x) {
          const bool in = col[j] >= 0;
          sm[j * k + i] = in ? M[(int64_t)col[j] * k + i] : 0.0;
          sv[j * k + i] = in ? V[(int64_t)col[j] * k + i] : 0.0;
        }
      __syncthreads();
      int nrot = 0;
      bool big = false;
      // inner rounds: the blocks' own pairs (first round of a sweep), then the cross pairs
      // inner round 0: (0,1) (2,3); 1: (0,2) (1,3); 2: (0,3) (1,2) -- slot 0 takes the first pair
      for (int ir = round == 0 ? 0 : 1; ir < 3; ++ir) {
        const int p = ir == 0 ? 2 * slot : slot;
        const int q = ir == 0 ? 2 * slot + 1 : (ir == 1 ? slot + 2 : 3 - slot);
        double* pt = part + 6 * slot;
        if (col[p] >= 0 && col[q] >= 0) {
          if (jacobi_rotate_split(sm + p * k, sm + q * k, sv + p * k, sv + q * k, k, h, lane, pt, eps, tiny, &big,
                                  big2))
            ++nrot;
        } else {
          __syncthreads();   // the same barrier count as a rotating slot
        }
        __syncthreads();
      }
      if (h == 0 && lane == 0 && nrot) atomicAdd(&ws[sweep & 1], (unsigned long long)nrot);
      if (h == 0 && lane == 0 && big) atomicAdd(&ws[4 + (sweep & 1)], 1ull);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (col[j] >= 0)
          for (int i = threadIdx.x; i < k; i += blockDim.x) {
            M[(int64_t)col[j] * k + i] = sm[j * k + i];
            V[(int64_t)col[j] * k + i] = sv[j * k + i];
          }
      grid.sync();
    }
    const unsigned long long rot = *(volatile unsigned long long*)&ws[sweep & 1];
    const unsigned long long nbig = *(volatile unsigned long long*)&ws[4 + (sweep & 1)];
    grid.sync();
    if (blockIdx.x == 0 && threadIdx.x == 0) ws[3] = (unsigned long long)(sweep + 1);
    // converged: no rotation, or only rotations below sqrt(big2) relative, after which the
    // off-diagonal products are O(big2) = O(eps / k) (quadratic convergence), so the next
    // sweep would find nothing above eps
    if (rot == 0 || nbig == 0) break;
  }
}

// ---------------------------------------------------------------- FP32 sweeps
// State of one factorisation in device memory.
struct SvdState {
  unsigned long long maxbits;    // largest |M_ij| (bits of a double)
  unsigned cnt[3];               // finished blocks of k_svd_angles, per step
  unsigned bad[3];               // pairs whose angle is not small
  unsigned long long cos2[3];    // largest cos^2 (bits of a double)
  double s2[3];                  // ||S||_F^2
  int skip_gram[4];              // step i: skip everything / only the update / S^2 / the fourth-order terms
  int skip_apply[3];
  int skip_s2[3];
  int skip_q[3];
  int done;                      // converged: the FP64 sweeps are skipped
  unsigned sweep_rot[2], sweep_big[2];
};

// the power of two that brings the largest element to [1, 2) (near the ends of FP64: as close as a power
// of two gets)
__device__ __forceinline__ double unit_scale(unsigned long long maxbits) {
  const int e = (int)(maxbits >> 52);
  return maxbits == 0 || e == 0x7FF ? 1.0 : __longlong_as_double((long long)max(2046 - e, 1) << 52);
}

__global__ void k_svd_max(const double* M, int64_t n, SvdState* st) {
  unsigned long long m = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    m = max(m, (unsigned long long)__double_as_longlong(fabs(M[e])));
  for (int o = 16; o; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (threadIdx.x % 32 == 0) atomicMax(&st->maxbits, m);
}

// A rotation in double-float: c = ch + cl, s = sh + sl (sh = 0: none).
struct __align__(16) Rot {
  float ch, cl, sh, sl;
};

// Rotates the FP32 columns (mp, mq) by one warp and returns the rotation. np, nq: squared norms, kept
// up to date. big: |cos| was above 3e-5, so another sweep is needed.
__device__ __forceinline__ Rot rotate32(float* mp, float* mq, int k, int lane, float& np, float& nq, float tol, float tiny,
                                        bool& big) {
  float ga = 0.f;
  for (int i = lane; i < k; i += 32) ga = fmaf(mp[i], mq[i], ga);
#pragma unroll
  for (int o = 16; o; o >>= 1) ga += __shfl_xor_sync(0xffffffffu, ga, o);
  const float den = sqrtf(np) * sqrtf(nq);
  if (!(fabsf(ga) > tol * den) || fminf(np, nq) <= tiny) return Rot{1.f, 0.f, 0.f, 0.f};
  const float z = (nq - np) / (2.f * ga), az = fabsf(z);
  const float t = copysignf(az > 1e9f ? 0.5f / az : 1.f / (az + sqrtf(fmaf(z, z, 1.f))), z);
  // c = 1 / sqrt(1 + t^2) to double-float: the FP32 value and one Newton correction; s = t c
  const float t2 = t * t, t2l = fmaf(t, t, -t2), w = 1.f + t2, wl = (t2 - (w - 1.f)) + t2l;
  const float c0 = rsqrtf(w), q = c0 * c0, ql = fmaf(c0, c0, -q), p = q * w, pl = fmaf(q, w, -p);
  const float e = ((1.f - p) - pl) - fmaf(q, wl, ql * w);
  const float cc = 0.5f * c0 * e;
  Rot r;
  r.ch = c0 + cc;
  r.cl = cc - (r.ch - c0);
  r.sh = t * r.ch;
  r.sl = fmaf(t, r.ch, -r.sh) + t * r.cl;
  for (int i = lane; i < k; i += 32) {
    const float x = mp[i], y = mq[i];
    mp[i] = fmaf(r.ch, x, -r.sh * y);
    mq[i] = fmaf(r.sh, x, r.ch * y);
  }
  np = fmaxf(np - t * ga, 0.f);
  nq = nq + t * ga;
  big = big || fabsf(ga) > 3e-5f * den;
  return r;
}

// (x, y) <- (c x - s y, s x + c y) for double-float x, y
__device__ __forceinline__ void rotate_df(const Rot& r, float& xh, float& xl, float& yh, float& yl) {
  float nh, nl;
  {
    const float a = r.ch * xh, ae = fmaf(r.ch, xh, -a), b = -r.sh * yh, be = fmaf(-r.sh, yh, -b);
    const float z = a + b, v = z - a, er = (a - (z - v)) + (b - v);
    const float lo = er + ae + be + (fmaf(r.ch, xl, r.cl * xh) - fmaf(r.sh, yl, r.sl * yh));
    nh = z + lo;
    nl = lo - (nh - z);
  }
  const float a = r.sh * xh, ae = fmaf(r.sh, xh, -a), b = r.ch * yh, be = fmaf(r.ch, yh, -b);
  const float z = a + b, v = z - a, er = (a - (z - v)) + (b - v);
  const float lo = er + ae + be + (fmaf(r.sh, xl, r.sl * xh) + fmaf(r.ch, yl, r.cl * yh));
  yh = z + lo;
  yl = lo - (yh - z);
  xh = nh;
  xl = nl;
}

constexpr int J32_MAX_SWEEPS = 14;
// squared norms below 1e-30 of the whole carry no resolvable direction (as in FP64)
__device__ __forceinline__ float tiny32(float fro2) { return 1e-30f * fro2; }

// One CTA, everything in shared memory (12 k^2 bytes): k <= J32_ONE. One warp per pair.
constexpr int J32_ONE = 72;
__global__ void __launch_bounds__(1024) k_jacobi32(const double* M, int k, SvdState* st, double* V0) {
  extern __shared__ float sj[];
  const int ld = k | 1, kk = k + (k & 1);
  float *m = sj, *vh = m + k * ld, *vl = vh + k * ld, *nrm = vl + k * ld;
  __shared__ int any, big;
  __shared__ float fro2;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32, nw = blockDim.x / 32;
  const double sc = unit_scale(st->maxbits);
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) {
    const int j = e / k, i = e % k;
    m[j * ld + i] = (float)(M[e] * sc);
    vh[j * ld + i] = i == j ? 1.f : 0.f;
    vl[j * ld + i] = 0.f;
  }
  __syncthreads();
  const float tol = 6e-8f * sqrtf((float)k);
  for (int sweep = 0; sweep < J32_MAX_SWEEPS; ++sweep) {
    for (int j = warp; j < k; j += nw) {   // fresh squared norms
      float s = 0.f;
      for (int i = lane; i < k; i += 32) s = fmaf(m[j * ld + i], m[j * ld + i], s);
      for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) nrm[j] = s;
    }
    if (threadIdx.x == 0) any = big = 0;
    __syncthreads();
    if (sweep == 0 && warp == 0) {
      float f = 0.f;
      for (int j = lane; j < k; j += 32) f += nrm[j];
      for (int o = 16; o; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
      if (lane == 0) fro2 = f;
    }
    __syncthreads();
    const float tiny = tiny32(fro2);
    for (int round = 0; round < kk - 1; ++round) {
      for (int pr = warp; pr < kk / 2; pr += nw) {
        const int a = rr_player(pr, round, kk), b = rr_player(kk - 1 - pr, round, kk);
        const int p = min(a, b), q = max(a, b);
        if (q >= k) continue;
        float np = nrm[p], nq = nrm[q];
        bool large = false;
        const Rot r = rotate32(m + p * ld, m + q * ld, k, lane, np, nq, tol, tiny, large);
        if (r.sh == 0.f) continue;
        for (int i = lane; i < k; i += 32) rotate_df(r, vh[p * ld + i], vl[p * ld + i], vh[q * ld + i], vl[q * ld + i]);
        if (lane == 0) {
          nrm[p] = np;
          nrm[q] = nq;
          any = 1;
          if (large) big = 1;
        }
      }
      __syncthreads();
    }
    const bool stop = !any || !big;
    __syncthreads();
    if (stop) break;
  }
  for (int e = threadIdx.x; e < k * k; e += blockDim.x) V0[e] = (double)vh[(e / k) * ld + e % k] + (double)vl[(e / k) * ld + e % k];
}

// The whole GPU (cooperative launch). The first nm CTAs hold M: block b is columns 8 b .. 8 b + 7, and
// a CTA takes two blocks per round to shared memory and rotates their 64 cross pairs, eight at a time,
// one warp each, after the pairs inside each block in the first round of a sweep. The other CTAs hold
// rows of V in shared memory throughout and apply the rotations of the round before, read from a list
// (rotations act on the rows of V independently): the double-float updates of V are three quarters of
// the arithmetic, and this way they run beside the FP32 sweeps on the SMs those leave idle. One grid
// barrier per round. Measured at k = 510: V beside M in the same 32 CTAs 15.8 ms, on its own CTAs
// 10.2 ms (the FP64 method 56 ms).
constexpr int J32_B = 8;
constexpr int J32_INNER = 2 * J32_B - 1;   // inner rounds of a round, the in-block pairs of round 0 first
struct J32Args {
  const double* M;
  int k, nm;             // columns, CTAs that hold M
  float *A, *nrm;        // FP32 copy of M and squared column norms, between rounds
  Rot* list;             // [2][J32_INNER][8 nm]
  SvdState* st;
  double* V0;
};
// columns of the pair that warp w of M-CTA c rotates in inner round ir
__device__ __forceinline__ void j32_pair(int c, int w, int round, int ir, int nbe, int& p, int& q) {
  const int ba = rr_player(c, round, nbe), bb = rr_player(nbe - 1 - c, round, nbe);
  if (ir < J32_B - 1) {   // inside the blocks: four warps each
    const int b = w < J32_B / 2 ? ba : bb, x = w % (J32_B / 2);
    const int u = rr_player(x, ir, J32_B), v = rr_player(J32_B - 1 - x, ir, J32_B);
    p = b * J32_B + min(u, v);
    q = b * J32_B + max(u, v);
  } else {
    p = ba * J32_B + w;
    q = bb * J32_B + (w + ir) % J32_B;
  }
}
__global__ void __launch_bounds__(32 * J32_B) k_jacobi32_blk(J32Args g) {
  namespace cg = cooperative_groups;
  cg::grid_group grid = cg::this_grid();
  extern __shared__ float sj[];
  const int k = g.k, ld = k | 1;
  const int lane = threadIdx.x % 32, warp = threadIdx.x / 32;
  const int nb = (k + J32_B - 1) / J32_B, nbe = nb + (nb & 1), npair = g.nm * J32_B;
  const bool on_m = (int)blockIdx.x < g.nm;
  // V rows of this CTA
  const int nv = (int)gridDim.x - g.nm, rows = (k + nv - 1) / nv, r0 = ((int)blockIdx.x - g.nm) * rows;
  const int nr = on_m ? 0 : max(0, min(rows, k - r0));
  float *m = sj, *ns = m + 2 * J32_B * ld;     // M-CTA: two blocks of columns, their norms
  float *vh = sj, *vl = vh + rows * ld;        // V-CTA
  {
    const double sc = unit_scale(g.st->maxbits);
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)k * k; e += (int64_t)gridDim.x * blockDim.x)
      g.A[e] = (float)(g.M[e] * sc);
    for (int e = threadIdx.x; e < nr * k; e += blockDim.x) {
      vh[e / k * ld + e % k] = r0 + e / k == e % k ? 1.f : 0.f;
      vl[e / k * ld + e % k] = 0.f;
    }
  }
  grid.sync();
  // the rotations of one round, inner rounds in order, applied to this CTA's rows
  auto apply = [&](int round, int buf) {
    const Rot* l = g.list + (int64_t)buf * J32_INNER * npair;
    auto one = [&](float4 f, int ir, int pr) {
      if (f.z == 0.f) return;
      int p, q;
      j32_pair(pr / J32_B, pr % J32_B, round, ir, nbe, p, q);
      const Rot r{f.x, f.y, f.z, f.w};
      for (int i = 0; i < nr; ++i) rotate_df(r, vh[i * ld + p], vl[i * ld + p], vh[i * ld + q], vl[i * ld + q]);
    };
    const int pr0 = threadIdx.x;
    for (int h = round == 0 ? 0 : 1; h < 2; ++h) {   // in-block pairs, cross pairs: their rotations loaded at once
      const int i0 = h ? J32_B - 1 : 0, n = h ? J32_B : J32_B - 1;
      float4 f[J32_B];
#pragma unroll
      for (int i = 0; i < J32_B; ++i)
        f[i] = i < n && pr0 < npair ? __ldcg((const float4*)(l + (int64_t)(i0 + i) * npair + pr0)) : make_float4(1.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int i = 0; i < J32_B; ++i) {
        if (i >= n) break;
        one(f[i], i0 + i, pr0);
        for (int pr = pr0 + (int)blockDim.x; pr < npair; pr += blockDim.x)
          one(__ldcg((const float4*)(l + (int64_t)(i0 + i) * npair + pr)), i0 + i, pr);
        __syncthreads();
      }
    }
  };
  // elements are in units of the largest, so the squared Frobenius norm is at least 1
  const float tiny = tiny32(1.f), tol = 6e-8f * sqrtf((float)k);
  int buf = 0, last = -1;   // list written this round; round whose list is still to be applied
  for (int sweep = 0; sweep < J32_MAX_SWEEPS; ++sweep) {
    for (int round = 0; round < nbe - 1; ++round, buf ^= 1) {
      if (round == 1 && blockIdx.x == 0 && threadIdx.x == 0)
        g.st->sweep_rot[(sweep + 1) & 1] = g.st->sweep_big[(sweep + 1) & 1] = 0;
      if (!on_m) {
        if (last >= 0) apply(last, buf ^ 1);
      } else {
        const int blk[2] = {rr_player((int)blockIdx.x, round, nbe), rr_player(nbe - 1 - (int)blockIdx.x, round, nbe)};
        for (int j = warp; j < 2 * J32_B; j += J32_B) {
          const int col = blk[j / J32_B] * J32_B + j % J32_B;
          if (col >= k) continue;
          float s = 0.f;
          for (int i = lane; i < k; i += 32) {
            const float x = __ldcg(g.A + (int64_t)col * k + i);
            m[j * ld + i] = x;
            s = fmaf(x, x, s);
          }
          if (round == 0) {   // fresh squared norms once per sweep
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) ns[j] = s;
          } else if (lane == 0) {
            ns[j] = __ldcg(g.nrm + col);
          }
        }
        __syncthreads();
        bool rot = false, big = false;
        for (int ir = round == 0 ? 0 : J32_B - 1; ir < J32_INNER; ++ir) {
          int p, q;
          j32_pair((int)blockIdx.x, warp, round, ir, nbe, p, q);
          Rot r{1.f, 0.f, 0.f, 0.f};
          if (p < k && q < k) {   // local columns: block 0 first
            const int lp = (p / J32_B == blk[0] ? 0 : J32_B) + p % J32_B, lq = (q / J32_B == blk[0] ? 0 : J32_B) + q % J32_B;
            float np = ns[lp], nq = ns[lq];
            r = rotate32(m + lp * ld, m + lq * ld, k, lane, np, nq, tol, tiny, big);
            if (r.sh != 0.f) {
              rot = true;
              if (lane == 0) {
                ns[lp] = np;
                ns[lq] = nq;
              }
            }
          }
          if (lane == 0) __stcg((float4*)(g.list + ((int64_t)buf * J32_INNER + ir) * npair + blockIdx.x * J32_B + warp),
                                make_float4(r.ch, r.cl, r.sh, r.sl));
          __syncthreads();
        }
        if (lane == 0 && rot) atomicAdd(&g.st->sweep_rot[sweep & 1], 1u);
        if (lane == 0 && big) atomicAdd(&g.st->sweep_big[sweep & 1], 1u);
        for (int j = warp; j < 2 * J32_B; j += J32_B) {
          const int col = blk[j / J32_B] * J32_B + j % J32_B;
          if (col >= k) continue;
          for (int i = lane; i < k; i += 32) __stcg(g.A + (int64_t)col * k + i, m[j * ld + i]);
          if (lane == 0) __stcg(g.nrm + col, ns[j]);
        }
      }
      last = round;
      grid.sync();
    }
    // the counters of this sweep are cleared two barriers later at the earliest: all CTAs read the same
    const unsigned rot = *(volatile unsigned*)&g.st->sweep_rot[sweep & 1], big = *(volatile unsigned*)&g.st->sweep_big[sweep & 1];
    if (rot == 0 || big == 0) break;
  }
  if (!on_m && last >= 0) apply(last, buf ^ 1);
  for (int e = threadIdx.x; e < nr * k; e += blockDim.x) {
    const int i = e % nr, j = e / nr;
    g.V0[(int64_t)j * k + r0 + i] = (double)vh[i * ld + j] + (double)vl[i * ld + j];
  }
}

// ---------------------------------------------------------------- FP64 refinement
// G <- 3/2 - G / 2, and M to unit scale: the angles' test below and that of k_jacobi_svd_blk take fourth
// powers of the elements, which leave FP64's range for elements beyond 1e+-77 (every pair then passed
// for orthogonal). A power of two changes no rounding; k_svd_emit puts it back on the singular values.
__global__ void k_svd_schulz(double* G, double* M, int k, const SvdState* st) {
  const double sc = unit_scale(st->maxbits);
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)k * k; e += (int64_t)gridDim.x * blockDim.x) {
    G[e] = (e / k == e % k ? 1.5 : 0.0) - 0.5 * G[e];
    M[e] *= sc;
  }
}

// S from G = M^T M (step `it`): S_pq = tan of the Jacobi angle for p < q, S_qp = -S_pq. Pairs that
// are orthogonal to eps, or whose smaller norm is negligible, stay; an angle above 0.1 is left to the
// FP64 sweeps. The last block decides how the step goes on.
__global__ void __launch_bounds__(256) k_svd_angles(const double* G, double* S, int k, double eps, double big2, SvdState* st, int it) {
  if (st->skip_gram[it]) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      st->skip_apply[it] = st->skip_s2[it] = st->skip_q[it] = 1;
      st->skip_gram[it + 1] = 1;
    }
    return;
  }
  __shared__ double tr;
  if (threadIdx.x < 32) {
    double f = 0;
    for (int j = threadIdx.x; j < k; j += 32) f += G[(int64_t)j * k + j];
    for (int o = 16; o; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    if (threadIdx.x == 0) tr = f;
  }
  __syncthreads();
  const double tiny = 1e-30 * tr;
  double mc = 0, s2 = 0;
  unsigned bad = 0;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)k * k; e += (int64_t)gridDim.x * blockDim.x) {
    const int q = (int)(e / k), p = (int)(e % k);   // S(p, q) at q k + p
    if (p > q) continue;
    double t = 0.0;
    if (p < q) {
      const double al = G[(int64_t)p * k + p], be = G[(int64_t)q * k + q], ga = G[e], ab = al * be;
      if (fmin(al, be) > tiny && ga * ga > eps * eps * ab) {
        const double d = be - al, g2 = 2.0 * ga;
        t = (d >= 0 ? g2 : -g2) / (fabs(d) + sqrt(fma(d, d, g2 * g2)));
        mc = fmax(mc, ga * ga / ab);
        if (!(fabs(t) <= 0.1)) {
          t = 0.0;
          ++bad;
        }
        s2 = fma(2.0 * t, t, s2);
      }
    }
    S[e] = t;
    S[(int64_t)p * k + q] = -t;
  }
  for (int o = 16; o; o >>= 1) {
    mc = fmax(mc, __shfl_xor_sync(0xffffffffu, mc, o));
    s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    bad += __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (threadIdx.x % 32 == 0) {
    atomicMax(&st->cos2[it], (unsigned long long)__double_as_longlong(mc));
    atomicAdd(&st->s2[it], s2);
    if (bad) atomicAdd(&st->bad[it], bad);
  }
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(&st->cnt[it], 1u) == gridDim.x - 1) {
    __threadfence();
    const double c2 = __longlong_as_double((long long)*(volatile unsigned long long*)&st->cos2[it]);
    const double n2 = *(volatile double*)&st->s2[it];
    const unsigned nbad = *(volatile unsigned*)&st->bad[it];
    // ||S||_F <= 1e-2 keeps the fourth-order exponential orthonormal to rounding
    const bool fine = n2 <= 1e-4;
    const bool conv = fine && nbad == 0 && c2 <= big2;
    st->skip_apply[it] = !fine || n2 == 0.0;
    st->skip_s2[it] = st->skip_apply[it] || n2 < 1e-16;
    st->skip_q[it] = st->skip_apply[it] || n2 < 1.6e-11;
    st->skip_gram[it + 1] = conv || !fine || nbad != 0;
    if (conv) st->done = 1;
  }
}

// P = S + S2 / 2 (in place of S), R = S / 6 + S2 / 24
__global__ void k_svd_series(double* S, const double* S2, double* R, int64_t n, const SvdState* st, int it) {
  if (st->skip_apply[it] || st->skip_s2[it]) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const double a = S[e], b = S2[e];
    S[e] = fma(0.5, b, a);
    R[e] = fma(1.0 / 24.0, b, a / 6.0);
  }
}

__global__ void k_svd_add2(double* M, const double* dM, double* V, const double* dV, int64_t n, const int* skip) {
  if (*skip) return;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    M[e] += dM[e];
    V[e] += dV[e];
  }
}

// ---------------------------------------------------------------- result
// norms of the columns of M, a warp each
__global__ void __launch_bounds__(256) k_svd_norms(const double* M, int k, double* sig) {
  const int j = blockIdx.x * 8 + threadIdx.x / 32, lane = threadIdx.x % 32;
  if (j >= k) return;
  double s = 0;
  for (int i = lane; i < k; i += 32) s = fma(M[(int64_t)j * k + i], M[(int64_t)j * k + i], s);
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) sig[j] = sqrt(s);
}

// Rank of a singular value: by bit pattern, a total order (NaN above infinity), so that the order below is
// a permutation whatever the input. Its entries index V (gather_cols_f64).
__device__ __forceinline__ unsigned long long order_key(double s) { return (unsigned long long)__double_as_longlong(fabs(s)); }

// U_j = m_j / sigma_j (0 when sigma_j is negligible), written in descending order of sigma (ties by
// index): sigma[rank], U[:, rank], order[rank] = original column. st: M is at unit scale (null: as
// given). One block per column.
__global__ void __launch_bounds__(128) k_svd_emit(const double* M, const double* sig, int k, double* U, double* sigma, int* order,
                                                  const SvdState* st) {
  const int j = blockIdx.x;
  const double sj = sig[j];
  const unsigned long long kj = order_key(sj);
  __shared__ int rk[4];
  __shared__ double fr[4];
  int r = 0;
  double f = 0;
  for (int i = threadIdx.x; i < k; i += 128) {
    const double s = sig[i];
    const unsigned long long ki = order_key(s);
    r += ki > kj || (ki == kj && i < j);
    f = fma(s, s, f);
  }
  for (int o = 16; o; o >>= 1) {
    r += __shfl_xor_sync(0xffffffffu, r, o);
    f += __shfl_xor_sync(0xffffffffu, f, o);
  }
  if (threadIdx.x % 32 == 0) {
    rk[threadIdx.x / 32] = r;
    fr[threadIdx.x / 32] = f;
  }
  __syncthreads();
  const int rank = rk[0] + rk[1] + rk[2] + rk[3];
  const double fro2 = fr[0] + fr[1] + fr[2] + fr[3];
  // columns at or below the Jacobi negligibility level were never orthogonalised: they get a zero
  // singular vector instead of a normalised rounding residue
  const double inv = (sj > 0 && sj * sj > 1e-30 * fro2) ? 1.0 / sj : 0.0;
  for (int i = threadIdx.x; i < k; i += 128) U[(int64_t)rank * k + i] = M[(int64_t)j * k + i] * inv;
  if (threadIdx.x == 0) {
    order[rank] = j;
    sigma[rank] = st ? sj / unit_scale(st->maxbits) : sj;
  }
}

int grid_of(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 4)); }

// co-resident blocks of a cooperative kernel
template <class K>
int resident(K kern, int threads, size_t smem) {
  int dev = 0, sms = 0, per = 0;
  FP_CUDA(cudaGetDevice(&dev));
  FP_CUDA(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  FP_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kern, threads, smem));
  return sms * per;
}

// FP64 sweeps from M and, unless init, the V given
void sweeps_f64(cudaStream_t s, double* Mat, int k, double* V, const int* skip, bool init, void* ws_dev) {
  if (k <= 32) {   // one CTA; above, its SM's FP64 pipe takes longer than the grid barriers (k = 64: 15 ms)
    // stopping rule |m_p.m_q| <= sqrt(k) eps |m_p||m_q|: a dot product of length k
    // carries rounding of that size, so a fixed 1e-15 could never be met
    k_jacobi_svd<<<1, 1024, 0, s>>>(Mat, V, k, 30, 1e-15 * sqrt((double)k), skip, init);
    FP_LAUNCH();
    return;
  }
  // one CTA per pair of two-column blocks, all co-resident (cooperative launch)
  const int nb = (k + 1) / 2, blocks = (nb + (nb & 1)) / 2;
  const size_t smem = (8 * (size_t)k + 12) * sizeof(double), most = (8 * 1024 + 12) * sizeof(double);
  static PerContext<int> per;
  const int max_blocks = per.get([&] {
    FP_CUDA(cudaFuncSetAttribute(k_jacobi_svd_blk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
    return resident(k_jacobi_svd_blk, JB_THREADS, most);
  });
  FP_CHECK(blocks <= max_blocks, FPEPS_ERR_CUDA, "svd: too few co-resident blocks");
  unsigned long long* ws = (unsigned long long*)ws_dev;
  int max_sweeps = 30;
  double eps = 1e-15 * sqrt((double)k);
  double big2 = eps / k;
  void* args[] = {&Mat, &V, &k, &max_sweeps, &eps, &big2, &skip, &init, &ws};
  count_launch();
  FP_CUDA(cudaLaunchCooperativeKernel((void*)k_jacobi_svd_blk, blocks, JB_THREADS, args, smem, s));
}

constexpr size_t kStateBytes = 512;
static_assert(sizeof(SvdState) <= kStateBytes && kStateBytes % sizeof(Rot) == 0, "state");
size_t list_bytes(int k) {
  const size_t nm = ((size_t)(k + J32_B - 1) / J32_B + 1) / 2;
  return k > J32_ONE ? 2 * J32_INNER * J32_B * nm * sizeof(Rot) : 0;
}

}  // namespace

// Up to this size the FP64 sweeps alone are as fast: the other way is ~30 launches.
constexpr int kDirect = 16;

size_t svd_work_bytes(int k) {
  const size_t kk = (size_t)k * k;
  if (k <= kDirect) return 0;
  return kStateBytes + list_bytes(k) + 3 * kk * sizeof(double) + (k > J32_ONE ? (kk + k) * sizeof(float) : 0);
}

void svd_jacobi_f64(cudaStream_t s, double* Mat, int k, double* U, double* sigma, double* V, int* order, void* ws_dev, void* work) {
  FP_CHECK(k <= 1024, FPEPS_ERR_UNSUPPORTED, "svd: k > 1024");
  ProfToken pt = prof_begin(PROF_FACTOR, s, 0.0, 16.0 * k * k);
  double* M = Mat;
  double* sig = (double*)((char*)ws_dev + 256);
  const SvdState* unit = nullptr;
  if (!work || k <= kDirect) {
    sweeps_f64(s, Mat, k, V, nullptr, true, ws_dev);
  } else {
    const int64_t kk = (int64_t)k * k;
    SvdState* st = (SvdState*)work;
    unit = st;
    // state, lists of rotations (16-byte entries), three matrices, the FP32 copy and norms
    double* T1 = (double*)((char*)work + kStateBytes + list_bytes(k));
    double *T2 = T1 + kk, *T3 = T2 + kk;
    FP_CUDA(cudaMemsetAsync(st, 0, sizeof(SvdState), s));
    k_svd_max<<<grid_of(kk), 256, 0, s>>>(Mat, kk, st);
    FP_LAUNCH();
    if (k <= J32_ONE) {
      static PerContext<bool> prepared;
      prepared.get([] {
        FP_CUDA(cudaFuncSetAttribute(k_jacobi32, cudaFuncAttributeMaxDynamicSharedMemorySize, (3 * J32_ONE * (J32_ONE + 1) + J32_ONE) * 4));
        return true;
      });
      k_jacobi32<<<1, 32 * std::min(32, (k + 1) / 2), (size_t)(3 * k * (k | 1) + k) * 4, s>>>(Mat, k, st, T1);
      FP_LAUNCH();
    } else {
      const int nb = (k + J32_B - 1) / J32_B, nm = (nb + (nb & 1)) / 2;
      auto smem_of = [](int n, int grid, int m_ctas) {
        const int rows = (n + grid - m_ctas - 1) / (grid - m_ctas);
        return (size_t)std::max(2 * J32_B * (n | 1) + 2 * J32_B, 2 * rows * (n | 1)) * 4;
      };
      static PerContext<int> per;
      const int max_blocks = per.get([&] {   // the largest need: 1024 columns on 64 + 64 CTAs
        const size_t most = smem_of(1024, 128, 64);
        FP_CUDA(cudaFuncSetAttribute(k_jacobi32_blk, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most));
        return std::min(resident(k_jacobi32_blk, 32 * J32_B, most), 152);
      });
      FP_CHECK(max_blocks >= 2 * nm, FPEPS_ERR_CUDA, "svd: too few co-resident blocks");
      const int blocks = std::min(max_blocks, nm + k);
      J32Args g;
      g.M = Mat;
      g.k = k;
      g.nm = nm;
      g.list = (Rot*)((char*)work + kStateBytes);
      g.A = (float*)(T3 + kk);
      g.nrm = g.A + kk;
      g.st = st;
      g.V0 = T1;
      void* args[] = {&g};
      count_launch();
      FP_CUDA(cudaLaunchCooperativeKernel((void*)k_jacobi32_blk, blocks, 32 * J32_B, args, smem_of(k, blocks, nm), s));
    }
    // column-major C = A B (or A^T B), optionally skipped or added to
    auto mul = [&](const double* A, bool ta, const double* B, double* C, double beta, const int* skip) {
      gemm_simt<double>(s, k, k, k, 1.0, A, ta ? k : 1, ta ? 1 : k, B, k, 1, beta, C, out_colmajor(k, k, k), skip, false);
    };
    mul(T1, true, T1, T2, 0.0, nullptr);
    k_svd_schulz<<<grid_of(kk), 256, 0, s>>>(T2, Mat, k, st);
    FP_LAUNCH();
    mul(T1, false, T2, V, 0.0, nullptr);
    mul(Mat, false, V, T3, 0.0, nullptr);
    M = T3;
    const double eps = 1e-15 * sqrt((double)k), big2 = eps / k;
    for (int it = 0; it < 3; ++it) {
      mul(M, true, M, T1, 0.0, &st->skip_gram[it]);
      k_svd_angles<<<grid_of(kk), 256, 0, s>>>(T1, T2, k, eps, big2, st, it);
      FP_LAUNCH();
      mul(T2, false, T2, T1, 0.0, &st->skip_s2[it]);
      k_svd_series<<<grid_of(kk), 256, 0, s>>>(T2, T1, Mat, kk, st, it);
      FP_LAUNCH();
      mul(T1, false, Mat, T2, 1.0, &st->skip_q[it]);
      mul(M, false, T2, T1, 0.0, &st->skip_apply[it]);
      mul(V, false, T2, Mat, 0.0, &st->skip_apply[it]);
      k_svd_add2<<<grid_of(kk), 256, 0, s>>>(M, T1, V, Mat, kk, &st->skip_apply[it]);
      FP_LAUNCH();
    }
    sweeps_f64(s, M, k, V, &st->done, false, ws_dev);
  }
  k_svd_norms<<<(k + 7) / 8, 256, 0, s>>>(M, k, sig);
  FP_LAUNCH();
  k_svd_emit<<<k, 128, 0, s>>>(M, sig, k, U, sigma, order, unit);
  FP_LAUNCH();
  prof_end(pt, s);
}

}  // namespace fpeps
