// Kernels that call the routines of small bonds alone (small_bond.cuh and the
// contraction of engine_kernels.cuh), compiled by test_gpu_small_bond_kernels.py
// for either CTA size (STN_CTA_THREADS).  All pointers are device memory; every
// launch is one CTA (check_keep: a warp, check_heads: one per element).
#include "engine_kernels.cuh"

STN_BEGIN

template <typename T, bool SM>
__global__ void __launch_bounds__(kThreads, 1) svd_kernel(int m, int n, const cplx<T> *A, cplx<T> *V, T *lam_out,
                                                          double cutoff, int kmax, void *gbuf, cplx<T> *vs,
                                                          cplx<T> *site, int *out, double *discarded, int truncate) {
  extern __shared__ __align__(16) char smem_raw[];
  double *red = reinterpret_cast<double *>(smem_raw), *disc = red + kRedDoubles;
  int *misc = reinterpret_cast<int *>(disc + 2), *perm = misc + 4;
  T *lam = reinterpret_cast<T *>(perm + kSmallSvdCols);
  char *u = reinterpret_cast<char *>(lam + kSmallSvdCols);
  if (tid() < 4) misc[tid()] = 0;
  if (tid() == 0) *disc = 0;
  __syncthreads();
  const Truncation<T> tr{perm, kmax, 0.0, misc, misc + 1, disc, vs, site};
  const int got = svd_small<T, SM>(m, n, A, V, truncate ? lam : lam_out, cutoff, SM ? u + 48 : gbuf, u, red,
                                   truncate ? &tr : nullptr);
  __syncthreads();
  if (truncate)
    for (int i = tid(); i < n; i += kThreads) lam_out[i] = lam[i];
  if (tid() == 0) {
    out[0] = got;
    out[1] = misc[0];
    *discarded = *disc;
  }
}

template <typename T, bool SM>
cudaError_t launch_svd(int m, int n, const void *A, void *V, void *lam, double cutoff, int kmax, void *gbuf, void *vs,
                       void *site, int *out, double *discarded, int truncate) {
  size_t smem = sizeof(double) * (kRedDoubles + 2) + sizeof(int) * (4 + kSmallSvdCols) + sizeof(T) * kSmallSvdCols + 48;
  if (SM) smem += 16 * static_cast<size_t>(n) * (m | 1);
  cudaError_t e = cudaFuncSetAttribute(svd_kernel<T, SM>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  svd_kernel<T, SM><<<1, kThreads, smem>>>(m, n, static_cast<const cplx<T> *>(A), static_cast<cplx<T> *>(V),
                                           static_cast<T *>(lam), cutoff, kmax, gbuf, static_cast<cplx<T> *>(vs),
                                           static_cast<cplx<T> *>(site), out, discarded, truncate);
  return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) gemm_kernel(int ta, int tb, int m, int n, int k, const cplx<T> *A, int lda,
                                                           const cplx<T> *B, int ldb, cplx<T> *C) {
  extern __shared__ __align__(16) char smem_raw[];
  cplx<T> *tile = reinterpret_cast<cplx<T> *>(smem_raw);
  tc_disable();
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  if (ta == 0 && tb == 0) cgemm<T, 0, 0>(m, n, k, one, A, lda, B, ldb, zero, C, n, tile);
  else if (ta == 0) cgemm<T, 0, 1>(m, n, k, one, A, lda, B, ldb, zero, C, n, tile);
  else cgemm<T, 1, 0>(m, n, k, one, A, lda, B, ldb, zero, C, n, tile);
}

template <typename T>
cudaError_t launch_gemm(int ta, int tb, int m, int n, int k, const void *A, const void *B, void *C) {
  const size_t smem = sizeof(cplx<T>) * kTileElems;
  gemm_kernel<T><<<1, kThreads, smem>>>(ta, tb, m, n, k, static_cast<const cplx<T> *>(A), ta ? m : k,
                                        static_cast<const cplx<T> *>(B), tb ? k : n, static_cast<cplx<T> *>(C));
  return cudaGetLastError();
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) qr_kernel(bool conj_t, int m, int n, const cplx<T> *A, cplx<T> *R,
                                                         cplx<T> *Q) {
  extern __shared__ __align__(16) char smem_raw[];
  qr_small<T>(m, n, A, conj_t ? m : n, conj_t, R, min(m, n), Q, reinterpret_cast<cplx<T> *>(smem_raw));
}

template <typename T>
cudaError_t launch_qr(int conj_t, int m, int n, const void *A, void *R, void *Q) {
  const size_t smem = sizeof(cplx<T>) * qr_small_elems(m, n, Q != nullptr);
  cudaError_t e = cudaFuncSetAttribute(qr_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  qr_kernel<T><<<1, kThreads, smem>>>(conj_t != 0, m, n, static_cast<const cplx<T> *>(A), static_cast<cplx<T> *>(R),
                                      static_cast<cplx<T> *>(Q));
  return cudaGetLastError();
}

template <typename T>
__global__ void keep_kernel(const T *lam, const int *perm, int n, int cap, double cutoff, double delta, int *out) {
  const int k = keep_count<T>(lam, perm, n, cap, cutoff, delta);
  if (threadIdx.x == 0) *out = k;
}

__device__ ff split(double x) {
  const float h = static_cast<float>(x);
  return ff_norm(ff{h, static_cast<float>(x - h)});
}
__device__ double joined(ff x) { return static_cast<double>(x.h) + x.l; }

__global__ void math_kernel(int what, int count, const double *x, double *y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  if (what == 0) y[i] = rsqrt64(x[i]);
  else if (what == 1) y[i] = reciprocal(x[i]);
  else if (what == 2) y[i] = joined(ff_rsqrt(split(x[i])));
  else y[i] = reciprocal(split(x[i]));
}

// in: re and im of x_j, ||x||^2; out: v0, gam, beta
__global__ void heads_kernel(int pairs, const double *in, double *out) {
  __shared__ cplx<double> d[3];
  __shared__ cplx<ff> f[3];
  const double *x = in + 3 * blockIdx.x;
  if (pairs) head_scaled(cmake<ff>(split(x[0]), split(x[1])), split(x[2]), f);
  else head_scaled(cmake<double>(x[0], x[1]), x[2], d);
  __syncwarp();
  if (threadIdx.x == 0)
    for (int i = 0; i < 3; ++i) {
      out[5 * blockIdx.x + 2 * i] = pairs ? joined(f[i].re) : d[i].re;
      if (i < 2) out[5 * blockIdx.x + 2 * i + 1] = pairs ? joined(f[i].im) : d[i].im;
    }
}

STN_END

extern "C" {
int check_svd(int precision, int shared, int m, int n, const void *A, void *V, void *lam, double cutoff, int kmax,
              void *gbuf, void *vs, void *site, int *out, double *discarded, int truncate) {
  using namespace stn;
  if (precision == 0)
    return shared ? launch_svd<double, true>(m, n, A, V, lam, cutoff, kmax, gbuf, vs, site, out, discarded, truncate)
                  : launch_svd<double, false>(m, n, A, V, lam, cutoff, kmax, gbuf, vs, site, out, discarded, truncate);
  return shared ? launch_svd<float, true>(m, n, A, V, lam, cutoff, kmax, gbuf, vs, site, out, discarded, truncate)
                : launch_svd<float, false>(m, n, A, V, lam, cutoff, kmax, gbuf, vs, site, out, discarded, truncate);
}
int check_gemm(int precision, int ta, int tb, int m, int n, int k, const void *A, const void *B, void *C) {
  return precision == 0 ? stn::launch_gemm<double>(ta, tb, m, n, k, A, B, C)
                        : stn::launch_gemm<float>(ta, tb, m, n, k, A, B, C);
}
int check_qr(int precision, int conj_t, int m, int n, const void *A, void *R, void *Q) {
  return precision == 0 ? stn::launch_qr<double>(conj_t, m, n, A, R, Q) : stn::launch_qr<float>(conj_t, m, n, A, R, Q);
}
int check_keep(int precision, const void *lam, const int *perm, int n, int cap, double cutoff, double delta, int *out) {
  if (precision == 0) stn::keep_kernel<double><<<1, 32>>>(static_cast<const double *>(lam), perm, n, cap, cutoff, delta, out);
  else stn::keep_kernel<float><<<1, 32>>>(static_cast<const float *>(lam), perm, n, cap, cutoff, delta, out);
  return cudaGetLastError();
}
int check_math(int what, int count, const double *x, double *y) {
  stn::math_kernel<<<(count + 255) / 256, 256>>>(what, count, x, y);
  return cudaGetLastError();
}
int check_heads(int pairs, int count, const double *in, double *out) {
  stn::heads_kernel<<<count, 32>>>(pairs, in, out);
  return cudaGetLastError();
}
}
