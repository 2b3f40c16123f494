// Internal declarations shared by the CUDA translation units of libfpeps.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>
#include <string>
#include <vector>

#include "context.cuh"
#include "fpeps.h"

namespace fpeps {

// ---------------------------------------------------------------- errors
struct Error {
  fpeps_status st;
  std::string msg;
};

#define FP_CUDA(call)                                                                  \
  do {                                                                                 \
    cudaError_t e_ = (call);                                                           \
    if (e_ != cudaSuccess)                                                             \
      throw ::fpeps::Error{FPEPS_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)}; \
  } while (0)

#define FP_CHECK(cond, code, text)                                   \
  do {                                                               \
    if (!(cond)) throw ::fpeps::Error{code, std::string(text)};      \
  } while (0)

// ---------------------------------------------------------------- launch accounting
// Every kernel launch of the library goes through FP_LAUNCH (count), and the
// hot kernel classes can be bracketed with CUDA events (prof_begin/prof_end)
// when profiling is enabled, so callers can time them on their own stream.
enum ProfKind {
  PROF_GEMM_TC = 0, PROF_GEMM_SIMT = 1, PROF_SANDWICH = 2, PROF_GRAM = 3, PROF_FACTOR = 4, PROF_SKETCH = 5, PROF_KINDS = 6
};
void count_launch();
struct ProfToken {
  int kind = -1;
  cudaEvent_t e0 = nullptr;
  double flops = 0, bytes = 0;
};
ProfToken prof_begin(int kind, cudaStream_t s, double flops, double bytes);
void prof_end(ProfToken& t, cudaStream_t s);

#define FP_LAUNCH()                  \
  do {                               \
    ::fpeps::count_launch();         \
    FP_CUDA(cudaGetLastError());     \
  } while (0)

// ---------------------------------------------------------------- memory
// Device memory owned through the env allocator. Arena buffers are released in
// bulk when the arena is reset.
struct Allocator {
  fpeps_allocator a{};
  bool has = false;
  cudaStream_t stream = nullptr;
  std::function<void()> reclaim;   // gives back what its owner can do without, before an allocation fails
  void* get(size_t bytes);
  void put(void* p);
};

struct Arena {
  Allocator* al = nullptr;
  std::vector<void*> live;
  void* get(size_t bytes) {
    void* p = al->get(bytes < 256 ? 256 : bytes);
    live.push_back(p);
    return p;
  }
  template <class T>
  T* get_n(size_t n) { return static_cast<T*>(get(n * sizeof(T))); }
  void reset() {
    for (void* p : live) al->put(p);
    live.clear();
  }
  ~Arena() { reset(); }
};

// ---------------------------------------------------------------- GEMM
// C(m,n) = alpha * sum_k A(m,k) B(n,k) + beta * C(m,n)
//   A(m,k) = A[m*a_m + k*a_k], B(n,k) = B[n*b_n + k*b_k]
//   addr(C(m,n)) = (m/mdiv)*c0 + (m%mdiv)*c1 + (n/ndiv)*c2 + (n%ndiv)*c3
struct OutMap {
  int64_t mdiv, c0, c1, ndiv, c2, c3;
};
inline OutMap out_rowmajor(int64_t M, int64_t N, int64_t ldc) { return OutMap{M, 0, ldc, N, 0, 1}; }
inline OutMap out_colmajor(int64_t M, int64_t N, int64_t ldc) { return OutMap{M, 0, 1, N, 0, ldc}; }

template <class T>
void gemm_simt(cudaStream_t s, int64_t M, int64_t N, int64_t K, T alpha, const T* A, int64_t a_m,
               int64_t a_k, const T* B, int64_t b_n, int64_t b_k, T beta, T* C, OutMap om,
               const int* skip = nullptr,    // device flag: nothing is done when it is set
               bool record = true);          // false: part of a step that has a profile record of its own

// Tensor-core GEMM for K-major A [M][lda] and B [N][ldb] (k contiguous), every operand split
// into two 11-bit halves: products that amortise it run on FP16 planes made beforehand (gemm_tc.cu),
// the others, and graded operands, split into TF32 on chip (gemm_onchip.cu).
//
// Grading, of a product on planes. Of the 256 terms of a row that share a scale, "tiny" ones are not zero
// and below 2^-17 of the largest (they lose bits), "large" ones at least 2^-9. Such a segment is deep
// when more than 24 terms are tiny, uneven when more than 17 are not large, narrow when less than 24 are
// large (fewer of each in a short segment). The sum of a deep segment that is not narrow, against one
// that is not uneven, is carried by large terms; of two that are not deep, by terms of 20 bits or more.
// So a product is graded, and left to the on-chip split, when an operand is deep somewhere and the
// other uneven somewhere, or a segment is both deep and narrow. N(0,1) data has one tiny term in 60000
// and one in 200 that is not large; rows times singular values, or blocks times small couplings, against
// such data are not graded.
// The words hold the mark of the last product that raised them, so a caller clears them once.
struct Grading {
  int deep[2], narrow, uneven[2];   // [2]: of A, of B
};
__device__ __forceinline__ bool is_graded(const Grading* g, int mark) {
  const volatile Grading* v = g;
  return v->narrow == mark || (v->deep[0] == mark && v->uneven[1] == mark) || (v->deep[1] == mark && v->uneven[0] == mark);
}
// The first 256 bytes of the scratch, cleared by the caller when it is new: the error word (set to 1
// when a bounded wait timed out), then a Grading. mark: not zero, another one for every product.
constexpr size_t kTcHeader = 256;
bool gemm_tc_supported(int64_t M, int64_t N, int64_t K, int64_t lda, int64_t ldb);
// Scratch of fewer bytes than gemm_tc_scratch_bytes, but at least gemm_onchip_scratch_bytes, sends the
// product to the on-chip split. settle: graded operands are recomputed on chip, decided on the device (three launches that return at
// once where there are none). Without it the caller looks at deep and narrow and calls gemm_tc_settle.
void gemm_tc(cudaStream_t s, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
             int64_t ldb, float* C, OutMap om, void* scratch, size_t scratch_bytes, int mark, bool settle = true);
void gemm_tc_settle(cudaStream_t s, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
                    int64_t ldb, float* C, OutMap om, void* scratch, size_t scratch_bytes, int mark);
size_t gemm_tc_scratch_bytes(int64_t M, int64_t N, int64_t K);
// hold_loads: self-test of the bounded waits (no loads issued); graded: nothing is done unless these
// operands are (null: always)
void gemm_onchip(cudaStream_t s, int64_t M, int64_t N, int64_t K, const float* A, int64_t lda, const float* B,
                 int64_t ldb, float* C, OutMap om, void* scratch, size_t scratch_bytes, bool hold_loads = false,
                 const Grading* graded = nullptr, int mark = 0);
size_t gemm_onchip_scratch_bytes(int64_t M, int64_t N, int64_t K);
// a split operand: planes [rows][k-blocks of 32 terms][32 hi, 32 lo halves], 2^-e of row r in the
// chunk c of 256 terms at inv[c * inv_stride + r]
struct SplitMat {
  const void* planes;
  const float* inv;
  int64_t inv_stride;
};
// self-test of the bounded waits of the planes kernel (no loads issued); planes: any device memory
void gemm_tc_hold(cudaStream_t s, int64_t M, int64_t N, int64_t K, void* planes, float* C, void* scratch);

// ---------------------------------------------------------------- sandwich
// Bundle order. A (ket, PEPO, bra) bundle of dims (n, nw, n) is indexed (x nw + x_w) n + x'
// everywhere except in the output of the sandwich, where the output bundle with unit stride
// (the one the next GEMM contracts over) is stored PEPO-index outermost, (x_w n + x) n + x':
// one output pair (v_w, z_w) then owns contiguous runs of n^2 elements. The operand that
// the next GEMM contracts with that bundle is stored in the same order (bundle_outer).
__host__ __device__ inline int64_t bundle_index(int x, int xw, int xp, int n, int nw, bool pepo_outer) {
  return pepo_outer ? ((int64_t)xw * n + x) * n + xp : ((int64_t)x * nw + xw) * n + xp;
}
// out[r][(x_w n + x) n + x'] = in[r][(x nw + x_w) n + x'] for r < rows
template <class T>
void bundle_outer(cudaStream_t s, const T* in, T* out, int64_t rows, int n, int nw);

// One orientation of the site sandwich: inputs legs (x, y) -> outputs (v, z).
struct SandOrient {
  int nx, nxw, ny, nyw, nv, nvw, nz, nzw, p;
  int nch;                 // nonzero PEPO channels
  const int* d_ch;         // [nch][4] = (xw, yw, vw, zw), sorted by (vw, zw)
  const int* d_pair_off;   // [nvw*nzw + 1] channel offsets per (vw, zw)
  const void* d_aw;        // [nch][nx][ny][nv][nz][p']  (A . W_ch)
  const void* d_ar;        // [nx][ny][nv][nz][p]        (A in these roles)
  int ch_host_max_per_pair;
  // tcgen05 sandwich (FP32 data): hi/lo operand images of A . W_ch and of the bra
  const void* d_kimg = nullptr;
  const void* d_arimg = nullptr;
};

template <class T>
void sandwich_apply(cudaStream_t s, const SandOrient& o, int64_t nt, int64_t nk, const T* in,
                    int64_t i_t, int64_t i_k, int64_t i_X, int64_t i_Y, T* out, int64_t o_t, int64_t o_k,
                    int64_t o_V, int64_t o_Z);

// 3xTF32 tensor-core version (mma.sync), float data; needs D <= 6 and D^2 p <= 144.
bool sandwich_mma_fits(const SandOrient& o);
void sandwich_apply_tc(cudaStream_t s, const SandOrient& o, int64_t nt, int64_t nk, const float* in, int64_t i_t,
                       int64_t i_k, int64_t i_X, int64_t i_Y, float* out, int64_t o_t, int64_t o_k, int64_t o_V,
                       int64_t o_Z);

// tcgen05 3xTF32 version (sandwich_tc.cu), float data; needs D <= 6, p <= 4 and p D^2 <= 144.
// The operand images are built once per site and orientation (sandwich_tc_images, sizes from
// sandwich_tc_image_floats); err is the tensor-core error word (set to 1 when a bounded wait
// timed out).
bool sandwich_tc_fits(const SandOrient& o);
void sandwich_tc_image_floats(const SandOrient& o, size_t* ket, size_t* bra);
void sandwich_tc_images(cudaStream_t s, const SandOrient& o, float* ket_img, float* bra_img);
void sandwich_apply_tcgen05(cudaStream_t s, const SandOrient& o, int64_t nt, int64_t nk, const float* in,
                            int64_t i_t, int64_t i_k, int64_t i_X, int64_t i_Y, float* out, int64_t o_t, int64_t o_k,
                            int64_t o_V, int64_t o_Z, int* err);

// Builds the role-permuted ket and the channel products A.W_ch for one orientation.
// roles[4] = leg index (0..3 = l,u,r,d) of (x, y, v, z).
template <class T>
void sandwich_prepare(cudaStream_t s, const T* A, const int dA[5], const T* W, const int dW[6], const int roles[4],
                      const int* d_ch, int nch, T* d_aw, T* d_ar);

// PEPO channel scan: flags[l,u,r,d] = 1 if block W[l,u,r,d,:,:] has a nonzero.
template <class T>
void pepo_scan(cudaStream_t s, const T* W, const int dW[6], int* d_flags);

// Row-0 boundary T[L][Dn][R] from the sandwich with the dimension-1 up legs.
template <class T>
void first_row_tensor(cudaStream_t s, const T* A, const int dA[5], const T* W, const int dW[6], T* out);

// ---------------------------------------------------------------- linalg
template <class T>
void gaussian_sketch(cudaStream_t s, T* out, int64_t n_rows, int64_t k, int64_t ld, const int64_t* perm_div,
                     uint64_t seed, uint64_t layer, uint64_t w2, uint64_t w3);

// upper triangle of G = Y^T Y (row-major), zeros below
template <class T>
void gram_f64(cudaStream_t s, const T* Y, int64_t m, int64_t k, int64_t ld, double* G);

// G (upper triangle of a Gram matrix, row-major, lower triangle zero) -> R with G = R^T R, and
// X = R^-T (row-major lower, i.e. R^-1 column-major); dependent columns give zero rows of R and zero
// rows and columns of X. info[0] |= 1 when a pivot is not finite.
void cholesky_inverse_f64(cudaStream_t s, double* G, double* X, int k, int* info);
// One-sided Jacobi SVD of the k x k col-major Mat (destroyed): Mat = U diag(sigma) V^T,
// sigma descending; U columns sorted, V columns in original order with order[rank] =
// original column. ws_dev: >= svd_ws_bytes(k) of device scratch; work: svd_work_bytes(k), or null
// (then FP64 sweeps alone).
inline size_t svd_ws_bytes(int k) { return 256 + 8 * (size_t)k; }
size_t svd_work_bytes(int k);
void svd_jacobi_f64(cudaStream_t s, double* Mat, int k, double* U, double* sigma, double* V, int* order,
                    void* ws_dev, void* work);

void gather_cols_f64(cudaStream_t s, const double* V, const int* order, int k, double* out);

template <class T>
void convert_f64(cudaStream_t s, const double* in, T* out, int64_t n);
template <class T>
void to_f64(cudaStream_t s, const T* in, double* out, int64_t n);

template <class T>
void frob_norm_f64(cudaStream_t s, const T* x, int64_t n, double* out);
template <class T>
void scale_by_inv(cudaStream_t s, T* x, int64_t n, const double* nrm);
// out[0] = <x, r> / <r, r> in FP64 (1 if that is not a positive finite number);
// out: >= 2 doubles of device memory
template <class T>
void scale_against(cudaStream_t s, const T* x, const T* r, int64_t n, double* out);

template <class T>
void permute3(cudaStream_t s, const T* in, T* out, int64_t d0, int64_t d1, int64_t d2, int p0, int p1, int p2);
// dst[c * ld_dst + r] = src[r * ld_src + c] for r < rows, c < cols; zero for rows <= r < ld_dst
template <class T>
void transpose_pad(cudaStream_t s, const T* src, int64_t rows, int64_t cols, int64_t ld_src, T* dst, int64_t ld_dst);
// out = a - b elementwise (out may alias a or b)
template <class T>
void sub_into(cudaStream_t s, T* out, const T* a, const T* b, int64_t n);
// out(i, j) += X(i, j) * R[j * k + j] for i < m, j < n (X, out column-major; R row-major FP64 k x k)
template <class T>
void add_diag_cols(cudaStream_t s, const T* X, int64_t m, int n, int64_t ldx, const double* R, int k, T* out,
                   int64_t ldo);
// A[j * ld + j] = 0 for j < k
template <class T>
void zero_diag(cudaStream_t s, T* A, int k, int64_t ld);
// dst (col-major rows x cols) = (T) src (row-major rows x cols)
template <class T>
void convert_f64_t(cudaStream_t s, const double* src, int64_t rows, int64_t cols, T* dst);

template <class T>
void fill(cudaStream_t s, T* x, int64_t n, T v);

template <class T>
void check_finite(cudaStream_t s, const T* x, int64_t n, int* flag);

}  // namespace fpeps
