#pragma once
// Dense routines of bonds that fit shared memory: the Householder QR of the
// sweeps and gauge steps (Sec. IV B).
// Included by engine_kernels.cuh, after its complex and warp helpers.
//
// At these sizes (a few to about a hundred columns) nothing is bound by a
// rate: a step is a chain of a reduction, a square root and a barrier, and on
// the FP64 side of the number of instructions, since a warp's FP64
// instruction takes 16 cycles of the SM's FP64 pipe (two FMAs a clock).  So a
// column belongs to a group of 8 lanes (three shuffle levels instead of
// five, and 8 rows per lane at 64 rows), only the warps that hold columns
// take part in a step's barrier, and square roots start from the hardware's
// approximation.

namespace stn {

constexpr int kGroup = 8;                       // lanes that share a column
constexpr int kGroups = kThreads / kGroup;      // columns in flight

// Barrier of the CTA's first nthr threads (a multiple of 32).
__device__ __forceinline__ void team_sync(int nthr) {
  if (nthr == 32) __syncwarp();
  else asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
}

// Threads of the team that holds `cols` columns, one per group.
__device__ __forceinline__ int team_threads(int cols) {
  return min(kThreads, (cols * kGroup + 31) & ~31);
}

// 1 / sqrt(x), x > 0: the hardware's approximation and one third-order
// (Halley) step, r + r e (1/2 + 3/8 e) with e = 1 - x r^2.
__device__ __forceinline__ double rsqrt64(double x) {
  double r;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x * r, r, 1.0);
  return fma(r * e, fma(0.375, e, 0.5), r);
}

template <typename S>
__device__ __forceinline__ S group_sum(S v) {
#pragma unroll
  for (int o = kGroup / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Reflector of x = col[j..m-1] with squared norm nx2 (P = I - 2 u u^dag, P x =
// gamma e_1, gamma = -(x_0 / |x_0|) ||x||) into u[j..m-1]; returns gamma.  One
// warp.
template <typename T>
__device__ __forceinline__ cplx<T> make_reflector(const cplx<T> *col, cplx<T> *u, int j, int m, double nx2) {
  const cplx<T> al = col[j];
  const double are = static_cast<double>(al.re), aim = static_cast<double>(al.im);
  const double a2 = are * are + aim * aim;
  const double nx = nx2 * rsqrt64(nx2);
  const bool zero = !(a2 > 1e-290);
  const double ra = rsqrt64(zero ? 1.0 : a2);
  const double pr = zero ? 1.0 : are * ra, pi = zero ? 0.0 : aim * ra;
  const double aa = zero ? 0.0 : a2 * ra;
  const cplx<T> gam = cmake<T>(static_cast<T>(-pr * nx), static_cast<T>(-pi * nx));
  const T sc = static_cast<T>(rsqrt64(2.0 * nx * (nx + aa)));
  for (int i = j + lane_id(); i < m; i += 32) {
    cplx<T> x = col[i];
    if (i == j) x = cmake<T>(x.re - gam.re, x.im - gam.im);
    u[i] = cscale(x, sc);
  }
  return gam;
}

// Householder QR in shared memory.  A is m x n: row-major with leading
// dimension lda (conj_t false), or given as its conjugate transpose, an n x m
// row-major array with leading dimension lda (conj_t true).  R (min(m, n) rows,
// zero below the diagonal, then zero rows up to r_rows) goes to Rout, row-major
// with leading dimension n; Rout may be A.  With Qout, the explicit Q (m x
// min(m, n)) goes there row-major, or with conj_t its conjugate transpose
// (min(m, n) x m); Qout may be A.  One barrier per column: the warp that holds
// column j + 1 applies reflector j to it and forms reflector j + 1 while the
// others still update theirs.  buf holds qr_small_elems elements.  CTA-wide.
//
// The blocked routine (qr_r_inplace) spends four barriers, two CTA
// reductions and a serial double-precision square root and division per
// column and reads its trailing columns from global memory.
__host__ __device__ __forceinline__ int64_t qr_small_elems(int m, int n, bool with_q) {
  const int64_t ld = m | 1;
  return ld * (n + (with_q ? (m < n ? m : n) : 2));
}

template <typename T>
static __device__ __noinline__ void qr_small(int m, int n, const cplx<T> *A, int lda, bool conj_t, cplx<T> *Rout,
                                             int r_rows, cplx<T> *Qout, cplx<T> *buf_) {
  const int ld = m | 1, steps = min(m, n);
  cplx<T> *Bm = in_smem<cplx<T>>(buf_), *U = Bm + n * ld;
  const bool keep = Qout != nullptr;
  for (int e = tid(); e < m * n; e += kThreads) {
    if (!conj_t) {
      const int i = e / n, c = e % n;
      Bm[c * ld + i] = A[i * lda + c];
    } else {
      const int c = e / m, i = e % m;
      Bm[c * ld + i] = cconj(A[c * lda + i]);
    }
  }
  __syncthreads();
  const int nthr = team_threads(n);
  const int gl = lane_id() & (kGroup - 1), g = tid() / kGroup;
  auto reflect = [&](int j) {
    cplx<T> *col = Bm + j * ld, *u = U + (keep ? j : (j & 1)) * ld;
    double s = 0;
    for (int i = j + lane_id(); i < m; i += 32) s += cabs2d(col[i]);
    s = warp_sum(s);
    cplx<T> gam = cmake<T>(0, 0);
    if (s > 1e-60) gam = make_reflector<T>(col, u, j, m, s);
    else  // (numerically) zero column: no reflector
      for (int i = j + lane_id(); i < m; i += 32) u[i] = cmake<T>(0, 0);
    __syncwarp();
    if (lane_id() == 0) col[j] = gam;
  };
  if (tid() < nthr) {
    if (warp_id() == 0) reflect(0);
    team_sync(nthr);
    for (int j = 0; j < steps; ++j) {
      const cplx<T> *u = U + (keep ? j : (j & 1)) * ld;
      const int i0 = j + ((gl - j) & (kGroup - 1));  // a lane keeps its rows: i = gl (mod 8)
      const int nxt = j + 1;
      for (int c = g; (c & ~3) < n; c += kGroups) {  // warp-uniform trip count
        const bool on = c > j && c < n;
        cplx<T> *b = Bm + min(c, n - 1) * ld;
        cplx<T> w = cmake<T>(0, 0);
        if (on)
#pragma unroll 4
          for (int i = i0; i < m; i += kGroup) cfma(w, cconj(u[i]), b[i]);
        w.re = group_sum(w.re);
        w.im = group_sum(w.im);
        if (on) {
          w = cmake<T>(T(-2) * w.re, T(-2) * w.im);
#pragma unroll 4
          for (int i = i0; i < m; i += kGroup) {
            cplx<T> x = b[i];
            cfma(x, u[i], w);
            b[i] = x;
          }
        }
        // the warp that has just brought column j + 1 up to date
        if (nxt < steps && (c & ~3) == (nxt & ~3)) {
          __syncwarp();
          reflect(nxt);
        }
      }
      team_sync(nthr);
    }
  }
  __syncthreads();
  for (int e = tid(); e < r_rows * n; e += kThreads) {
    const int i = e / n, c = e % n;
    Rout[e] = i < steps && c >= i ? Bm[c * ld + i] : cmake<T>(0, 0);
  }
  if (!keep) {
    __syncthreads();
    return;
  }
  __syncthreads();
  // Q e_c = P_0 ... P_c e_c (a reflector below row c leaves e_c alone)
  for (int c = g; (c & ~3) < steps; c += kGroups) {
    const int top = min(steps - 1, (c & ~3) + 3);  // largest column of the warp
    cplx<T> *q = Bm + min(c, steps - 1) * ld;
    const bool col = c < steps;
    if (col)
      for (int i = gl; i < m; i += kGroup) q[i] = cmake<T>(i == c ? T(1) : T(0), 0);
    for (int j = top; j >= 0; --j) {
      const cplx<T> *u = U + j * ld;
      const int i0 = j + ((gl - j) & (kGroup - 1));
      const bool on = col && j <= c;
      cplx<T> w = cmake<T>(0, 0);
      if (on)
#pragma unroll 4
        for (int i = i0; i < m; i += kGroup) cfma(w, cconj(u[i]), q[i]);
      w.re = group_sum(w.re);
      w.im = group_sum(w.im);
      if (on) {
        w = cmake<T>(T(-2) * w.re, T(-2) * w.im);
#pragma unroll 4
        for (int i = i0; i < m; i += kGroup) {
          cplx<T> x = q[i];
          cfma(x, u[i], w);
          q[i] = x;
        }
      }
    }
  }
  __syncthreads();
  for (int e = tid(); e < m * steps; e += kThreads) {
    if (!conj_t) {
      const int i = e / steps, c = e % steps;
      Qout[e] = Bm[c * ld + i];
    } else {
      const int c = e / m, i = e % m;
      Qout[e] = cconj(Bm[c * ld + i]);
    }
  }
  __syncthreads();
}

}  // namespace stn
