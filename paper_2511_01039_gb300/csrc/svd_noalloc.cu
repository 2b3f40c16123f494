// Scratch-free variant of the small FP64 SVD (fpeps_svd_f64): the same
// factorisation, with its working storage in a fixed device array
// instead of memory obtained from cudaMallocAsync.
//
// Who needs it: callers that must not allocate device memory at the moment
// they need the factorisation -- for example code running after a framework
// has reserved the whole device memory pool for its own allocator (so that
// cudaMallocAsync would fail or fight it), or a latency-critical loop in which
// an allocation could synchronise, fragment the pool or fail. They pass only
// their input and output buffers; this entry point allocates nothing.
//
// The working storage is g_svd_scratch below: 5 k^2 doubles (working matrix, accumulated
// rotations and the refinement's products), k^2 floats (the FP32 sweeps), lists of rotations,
// ordering, counters and norms, for k <= FPEPS_SVD_NOALLOC_MAX_K (256), about 3 MB. Every GPU that loads the
// library holds it until the process exits. In host code the symbol names a
// host-side stand-in, not device memory, so it is never handed to a kernel
// directly: on the first call in a context its device address is looked up with
// cudaGetSymbolAddress and kept for the later calls there (a context that follows
// a cudaDeviceReset looks it up again). All calls share the array: calls whose work overlaps on the GPU (different streams,
// or different host threads) race on it.
#include <exception>

#include "common.cuh"

namespace fpeps {
namespace {

constexpr int kMaxK = FPEPS_SVD_NOALLOC_MAX_K;
// two matrices, the factorisation's work (svd_work_bytes: three more, an FP32 copy and lists of rotations), order, counters and norms
constexpr size_t kScratchBytes = 5 * (size_t)kMaxK * kMaxK * sizeof(double) + ((size_t)kMaxK + 1) * kMaxK * sizeof(float) + 70000 +
                                 (size_t)kMaxK * (sizeof(int) + sizeof(double)) + 4096;
static __device__ __align__(256) unsigned char g_svd_scratch[kScratchBytes];

// device address of g_svd_scratch in the current context (looked up once)
char* scratch_address() {
  static PerContext<char*> per;
  return per.get([] {
    void* p = nullptr;
    FP_CUDA(cudaGetSymbolAddress(&p, g_svd_scratch));
    FP_CHECK(p != nullptr, FPEPS_ERR_CUDA, "cudaGetSymbolAddress returned NULL");
    return static_cast<char*>(p);
  });
}

}  // namespace
}  // namespace fpeps

extern "C" fpeps_status fpeps_svd_f64_noalloc(const double* M, int32_t k, double* U, double* sigma, double* V,
                                              void* cuda_stream) {
  try {
    if (!M || !U || !sigma || !V || k < 1) throw fpeps::Error{FPEPS_ERR_ARG, "bad SVD arguments"};
    if (k > fpeps::kMaxK)
      throw fpeps::Error{FPEPS_ERR_ARG, "k exceeds FPEPS_SVD_NOALLOC_MAX_K (256): use fpeps_svd_f64"};
    cudaStream_t s = (cudaStream_t)cuda_stream;
    char* scr = fpeps::scratch_address();
    const size_t kk = (size_t)k * k;
    double* Mw = reinterpret_cast<double*>(scr);
    double* Vw = Mw + kk;
    char* work = reinterpret_cast<char*>(Vw + kk);   // 256-byte aligned regions from here on
    auto up = [](size_t b) { return (b + 255) / 256 * 256; };
    work = scr + up((size_t)(work - scr));
    char* ws = work + up(fpeps::svd_work_bytes(k));
    int* order = reinterpret_cast<int*>(ws + up(fpeps::svd_ws_bytes(k)));
    if (reinterpret_cast<char*>(order + k) > scr + fpeps::kScratchBytes)
      throw fpeps::Error{FPEPS_ERR_ARG, "svd scratch too small"};
    // every region is rewritten before it is read: Mw by this copy, the rest by the
    // factorisation (which clears its counters on entry)
    FP_CUDA(cudaMemcpyAsync(Mw, M, kk * sizeof(double), cudaMemcpyDeviceToDevice, s));
    fpeps::svd_jacobi_f64(s, Mw, k, U, sigma, Vw, order, ws, work);
    fpeps::gather_cols_f64(s, Vw, order, k, V);
    FP_CUDA(cudaStreamSynchronize(s));
    return FPEPS_OK;
  } catch (const fpeps::Error& e) {
    return e.st;
  } catch (const std::exception&) {
    return FPEPS_ERR_ARG;
  }
}
