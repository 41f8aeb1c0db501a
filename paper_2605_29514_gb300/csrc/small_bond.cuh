#pragma once
// Dense routines of bonds that fit shared memory: the Householder QR of the
// sweeps and gauge steps, and the SVD of the truncation (Sec. IV B, Eq. 8).
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
constexpr int kSmallSvdCols = 128;              // column indices fit the 7 low bits of a pivot key

// Barrier of the CTA's first nthr threads (a multiple of 32).
__device__ __forceinline__ void team_sync(int nthr) {
  if (nthr == 32) __syncwarp();
  else asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
}

// The same barrier with an OR over its threads.
__device__ __forceinline__ bool team_any(int nthr, bool v) {
  if (nthr == 32) return __any_sync(0xffffffffu, v);
  int r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.s32 p, %1, 0;\n\t"
      "barrier.cta.red.or.pred q, 1, %2, p;\n\t"
      "selp.s32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"(v ? 1 : 0), "r"(nthr)
      : "memory");
  return r != 0;
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

// SVD of a bond in double precision, in shared memory: Householder QR with
// column pivoting, then one-sided (Hestenes) Jacobi on the rows of R, the
// preconditioning of Drmac and Veselic (SIAM J. Matrix Anal. Appl. 29, 2008).
// A (m x n, row-major, leading dimension n) = Q R, R in the original column
// order; rotating the rows of R until they are orthogonal gives the rows
// sigma_i v_i^dag, so no rotation is accumulated.  lam[i] = sigma_i^2 (unsorted,
// zero beyond the numerical rank, which is returned) and column i of V (n x n,
// column-major; columns beyond the rank are not written, except column 0 of a
// zero matrix) = v_i.  Values that are not finite give lam = NaN.
//
// Against Jacobi on A's columns with accumulated V (what bonds that fit
// shared memory ran before) this takes about half the sweeps and a quarter of
// the rotations on the matrices of a d = 3 and a d = 5 run, and rotates one
// matrix instead of two.  A group of 8 lanes rotates a pair; the angle is
// found in single precision from exponent-scaled numbers, and the cosine,
// sine and phase are brought to double precision by a third-order correction,
// so the rotation is unitary to rounding and only its angle is approximate
// (which costs no sweep: an angle good to 1e-7 leaves 1e-7 of the product).
//
// cutoff > 0 (the truncation's): two rows whose norms are both so small that
// all such rows together stay below half of cutoff sigma_1 are not rotated
// against each other.  They are dropped whatever their mutual angles are, and
// the sum of their squares, the discarded weight, does not change.
//
// buf: n (m | 1) complex doubles; u: m of them; nr: n doubles (all shared
// memory); n <= kSmallSvdCols.  CTA-wide.
template <typename T>
static __device__ __noinline__ int svd_small(int m, int n, const cplx<T> *A, cplx<T> *V, T *lam, double cutoff,
                                             cplx<double> *buf_, cplx<double> *u_, double *nr_) {
  const int ld = m | 1, steps = min(m, n);
  cplx<double> *Bm = in_smem<cplx<double>>(buf_), *u = in_smem<cplx<double>>(u_);
  double *nr = in_smem<double>(nr_);
  for (int e = tid(); e < m * n; e += kThreads) {
    const int i = e / n, c = e % n;
    const cplx<T> x = A[e];
    Bm[c * ld + i] = cmake<double>(static_cast<double>(x.re), static_cast<double>(x.im));
  }
  __syncthreads();
  const int gl = lane_id() & (kGroup - 1), g = tid() / kGroup;
  constexpr double eps2 = 1.11e-16 * 1.11e-16;
  // largest of k numbers >= 0 (or -1) by their high words, column in the low
  // bits; every warp finds it by itself
  auto top_key = [&](int k) {
    int key = -1;
    for (int c = lane_id(); c < k; c += 32) {
      const int hi = __double2hiint(nr[c]);
      key = max(key, hi < 0 ? -1 : ((hi & ~127) | c));
    }
    return __reduce_max_sync(0xffffffffu, key);
  };
  int rank = 0;
  double neg = 0.0;  // squared norm of a negligible row
  bool finite = true;
  {
    const int nthr = team_threads(n);
    if (tid() < nthr) {
      for (int c = g; (c & ~3) < n; c += kGroups) {
        double s = 0;
        if (c < n)
          for (int i = gl; i < m; i += kGroup) s += cabs2(Bm[c * ld + i]);
        s = group_sum(s);
        if (gl == 0 && c < n) nr[c] = s <= 1.7e308 ? s : __longlong_as_double(0x7ff0000000000000ll);
      }
    }
    __syncthreads();
    const int k0 = top_key(n);
    finite = k0 < 0x7ff00000;
    neg = eps2 * nr[k0 & 127];
    __syncthreads();
    if (tid() < nthr && finite) {
      for (int j = 0; j < steps; ++j) {
        const int key = top_key(n);
        const int p = key & 127;
        const double nx2 = key < 0 ? 0.0 : nr[p];
        if (!(nx2 > neg)) break;  // the rest is below rounding (also: a zero matrix)
        if (warp_id() == (p & (kGroups - 1)) / 4) {
          cplx<double> *col = Bm + p * ld;
          const cplx<double> gam = make_reflector<double>(col, u, j, m, nx2);
          __syncwarp();
          for (int i = j + lane_id(); i < m; i += 32) col[i] = i == j ? gam : cmake<double>(0, 0);
        }
        team_sync(nthr);
        const int i0 = j + ((gl - j) & (kGroup - 1));
        for (int c = g; (c & ~3) < n; c += kGroups) {
          const bool on = c < n && c != p && nr[min(c, n - 1)] >= 0.0;
          cplx<double> *b = Bm + min(c, n - 1) * ld;
          cplx<double> w = cmake<double>(0, 0);
          if (on)
#pragma unroll 4
            for (int i = i0; i < m; i += kGroup) cfma(w, cconj(u[i]), b[i]);
          w.re = group_sum(w.re);
          w.im = group_sum(w.im);
          double s = 0;
          if (on) {
            w = cmake<double>(-2.0 * w.re, -2.0 * w.im);
#pragma unroll 4
            for (int i = i0; i < m; i += kGroup) {
              cplx<double> x = b[i];
              cfma(x, u[i], w);
              b[i] = x;
              if (i > j) s = fma(x.re, x.re, fma(x.im, x.im, s));
            }
          }
          s = group_sum(s);
          if (gl == 0 && c < n) {
            if (on) nr[c] = s;
            else if (c == p) nr[c] = -1.0;
          }
        }
        team_sync(nthr);
        rank = j + 1;
      }
    }
  }
  // the rank is known to the team's threads
  if (tid() == 0) reinterpret_cast<int *>(u)[0] = rank;
  __syncthreads();
  rank = reinterpret_cast<int *>(u)[0];
  __syncthreads();

  // rows of R: row i at Bm[c ld + i], ld odd, so 8 lanes over c meet no bank twice
  const int kk = rank + (rank & 1), half = kk / 2;
  const int nthr = team_threads(max(1, half));
  const double tol = 4.0 * 1.11e-16 * sqrt(static_cast<double>(n)), tol2 = tol * tol;
  auto norms = [&]() {
    for (int i = g; (i & ~3) < kk; i += nthr / kGroup) {
      double s = 0;
      if (i < rank)
        for (int c = gl; c < n; c += kGroup) s += cabs2(Bm[c * ld + i]);
      s = group_sum(s);
      if (gl == 0 && i < rank) nr[i] = s;
    }
  };
  if (tid() < nthr && finite) {
    for (int sweep = 0; sweep < kMaxSweepsD && rank > 1; ++sweep) {
      norms();
      team_sync(nthr);
      const double noise = cutoff * cutoff * nr[top_key(rank) & 127] / (4.0 * rank);
      team_sync(nthr);
      bool rotated = false;
      for (int round = 0; round < kk - 1; ++round) {
        for (int pi = g; (pi & ~3) < half; pi += nthr / kGroup) {
          int p, q;
          if (pi == 0) { p = kk - 1; q = round; }
          else { p = round + pi; q = round - pi; if (p >= kk - 1) p -= kk - 1; if (q < 0) q += kk - 1; }
          if (p > q) { const int t = p; p = q; q = t; }
          bool on = pi < half && q < rank;
          if (!on) p = q = 0;
          const double al = nr[p], be = nr[q];
          on = on && al > neg && be > neg && (al > noise || be > noise);
          cplx<double> dot = cmake<double>(0, 0);
          if (on)
#pragma unroll 4
            for (int c = gl; c < n; c += kGroup) cfma(dot, cconj(Bm[c * ld + p]), Bm[c * ld + q]);
          if (!__any_sync(0xffffffffu, on)) continue;
          dot.re = group_sum(dot.re);
          dot.im = group_sum(dot.im);
          if (!(cabs2(dot) > tol2 * al * be)) on = false;
          if (on) {
            rotated = true;
            // numbers scaled by a power of two so that the larger norm is in [1, 2)
            const int ex = max(1, __double2hiint(fmax(al, be)) >> 20);
            const double sc = __hiloint2double((2046 - min(2045, ex)) << 20, 0);
            const float df = static_cast<float>((be - al) * sc);
            const float gr = static_cast<float>(dot.re * sc), gi = static_cast<float>(dot.im * sc);
            const float mx = fmaxf(fmaxf(fabsf(gr), fabsf(gi)), 1e-37f), imx = 1.f / mx;
            const float ga = gr * imx, gb = gi * imx, g2 = ga * ga + gb * gb, gl2 = rsqrtf(g2);
            const float absg = mx * (g2 * gl2);
            const float zeta = df / (2.f * absg), az = fabsf(zeta);
            float tf = az > 1e10f ? 0.5f / az : 1.f / (az + sqrtf(1.f + az * az));
            if (zeta < 0.f) tf = -tf;
            const double t = static_cast<double>(tf), w = fma(t, t, 1.0);
            double cs = static_cast<double>(rsqrtf(fmaf(tf, tf, 1.f)));
            double d = fma(-w * cs, cs, 1.0);
            cs = fma(cs * d, fma(0.375, d, 0.5), cs);
            const double sn = t * cs;
            double ur = static_cast<double>(ga * gl2), ui = -static_cast<double>(gb * gl2);
            d = fma(-ur, ur, fma(-ui, ui, 1.0));
            d = fma(d, fma(0.375, d, 0.5), 1.0);
            const cplx<double> uc = cmake<double>(ur * d, ui * d);  // conj(g / |g|)
#pragma unroll 2
            for (int c = gl; c < n; c += kGroup) {
              const cplx<double> x = Bm[c * ld + p], y = cmul(uc, Bm[c * ld + q]);
              Bm[c * ld + p] = cmake<double>(fma(cs, x.re, -sn * y.re), fma(cs, x.im, -sn * y.im));
              Bm[c * ld + q] = cmake<double>(fma(sn, x.re, cs * y.re), fma(sn, x.im, cs * y.im));
            }
            if (gl == 0) {
              const double tg = t * static_cast<double>(absg) * __hiloint2double(min(2045, ex) << 20, 0);
              nr[p] = fmax(al - tg, 0.0);
              nr[q] = fmax(be + tg, 0.0);
            }
          }
        }
        team_sync(nthr);
      }
      if (!team_any(nthr, rotated)) break;
    }
    norms();
  }
  __syncthreads();
  for (int e = tid(); e < n * rank; e += kThreads) {
    const int i = e / n, c = e % n;
    const double s = nr[i];
    const cplx<double> x = Bm[c * ld + i];
    const double inv = s > 0.0 ? rsqrt64(s) : 0.0;
    V[e] = cmake<T>(static_cast<T>(x.re * inv), static_cast<T>(-x.im * inv));
  }
  if (rank == 0)
    for (int c = tid(); c < n; c += kThreads) V[c] = cmake<T>(c == 0 ? T(1) : T(0), 0);
  for (int i = tid(); i < n; i += kThreads)
    lam[i] = !finite ? static_cast<T>(__longlong_as_double(0x7ff8000000000000ll)) : i < rank ? static_cast<T>(nr[i]) : T(0);
  __syncthreads();
  return rank;
}

}  // namespace stn
