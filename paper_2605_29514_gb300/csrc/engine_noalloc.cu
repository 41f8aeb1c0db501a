#include "engine_kernels.cuh"

#include <mutex>

namespace stn {

// ---------------------------------------------------------------------------
// Allocation-free large-bond SVD.  Some callers cannot allocate device memory
// at the moment they need this routine: code running inside a host callback
// or under a framework's memory pool that forbids cudaMalloc mid-stream, or an
// embedded runtime that hands out only the buffers it owns.  For them the work
// copy of the input lives in this file-scope array instead of a buffer the
// caller or the library would allocate.  Every GPU that loads the library
// holds the array until the process exits.  All calls share it: it keeps the
// last call's contents, and two calls that overlap on the GPU (different
// streams, or different host threads on one stream without ordering) race
// on it.  Each call writes every scratch element it later reads, so nothing
// has to start at zero.
constexpr size_t kNoAllocScratchBytes = size_t(1) << 20;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) svd_noalloc_kernel(int m, int n, const cplx<T> *C,
                                                                  cplx<T> *work, cplx<T> *V, T *sig2) {
  extern __shared__ __align__(16) char smem_raw[];
  tc_disable();
  const DenseSmem s = dense_smem<T>(smem_raw);
  svd_bond<T, false>(m, n, C, work, V, sig2, reinterpret_cast<cplx<T> *>(s.buf), reinterpret_cast<cplx<T> *>(s.uv), s.red,
                     s.flag, s.rv_wrk);
}

size_t noalloc_scratch_bytes() { return kNoAllocScratchBytes; }

// Device address of the scratch array on the current device.  Host code may
// not pass g_noalloc_scratch itself: on the host that name is a stand-in, not
// a device address.  The address is looked up once per device, with that
// device current, on the first call made there.
static cudaError_t noalloc_scratch_ptr(void **out) {
  constexpr int kMaxDevices = 64;
  static std::mutex mu;
  static void *ptr[kMaxDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (ptr[dev] == nullptr) {
    void *p = nullptr;
    e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) return e;
    ptr[dev] = p;
  }
  *out = ptr[dev];
  return cudaSuccess;
}

template <typename T>
static cudaError_t launch_svd_noalloc_t(int m, int n, const void *C, void *V, void *sig2, cudaStream_t s) {
  void *work = nullptr;
  cudaError_t e = noalloc_scratch_ptr(&work);
  if (e != cudaSuccess) return e;
  if (shares_svd<T>(m, n))
    return launch_dense_shared<T>(true, m, n, const_cast<cplx<T> *>(static_cast<const cplx<T> *>(C)),
                                  static_cast<cplx<T> *>(work), static_cast<cplx<T> *>(V), static_cast<T *>(sig2), s);
  const size_t smem = dense_smem_bytes<T>();
  e = cudaFuncSetAttribute(svd_noalloc_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  svd_noalloc_kernel<T><<<1, kThreads, smem, s>>>(m, n, static_cast<const cplx<T> *>(C),
                                                  static_cast<cplx<T> *>(work), static_cast<cplx<T> *>(V),
                                                  static_cast<T *>(sig2));
  return cudaGetLastError();
}

cudaError_t launch_svd_noalloc(int precision, int m, int n, const void *C, void *V, void *sig2,
                               cudaStream_t s) {
  return precision == 0 ? launch_svd_noalloc_t<double>(m, n, C, V, sig2, s)
                        : launch_svd_noalloc_t<float>(m, n, C, V, sig2, s);
}

}  // namespace stn
