#pragma once
// Dense routines of bonds that fit shared memory: the Householder QR of the
// sweeps and gauge steps, and the SVD of the truncation (Sec. IV B, Eq. 8).
// Included by engine_kernels.cuh, after its complex and warp helpers.
//
// At these sizes (a few to about a hundred columns) nothing is bound by a
// rate: a step is a chain of a reduction, a square root and a barrier.  A
// column belongs to a group of 8 lanes (three shuffle levels instead of five),
// only the warps that hold columns take part in a step's barrier, and square
// roots start from the hardware's approximation.
//
// A double-precision operation takes 64 cycles, and an SM issues a warp's every
// 19 whatever its active lanes (measured; a dependent FP32 FMA takes 4.6), so the
// complex64 path computes what has to be better than single precision in pairs of
// floats (ff, 48 bits): its SVDs, and the norms and scalars of its reflectors.

STN_BEGIN

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

// ---------------------------------------------------------------------------
// Pairs of floats, value h + l with |l| <= ulp(h) / 2: the error-free sum and
// product of Knuth and Dekker (the product's error by FMA), about 2^-46
// relative per operation.  The intrinsics keep a product from being contracted
// into the sum that follows it.
struct ff {
  float h, l;
};
__device__ __forceinline__ ff ff_of(float x) { return ff{x, 0.f}; }
__device__ __forceinline__ ff ff_neg(ff a) { return ff{-a.h, -a.l}; }
// renormalises h + l with |l| well below |h|
__device__ __forceinline__ ff ff_norm(ff a) {
  const float s = __fadd_rn(a.h, a.l);
  return ff{s, __fsub_rn(a.l, __fsub_rn(s, a.h))};
}
// acc.h + x exactly into acc.h and (added to) acc.l; acc is renormalised later
__device__ __forceinline__ void ff_push(ff &acc, float x, float low) {
  const float s = __fadd_rn(acc.h, x), b = __fsub_rn(s, acc.h);
  const float e = __fadd_rn(__fsub_rn(acc.h, __fsub_rn(s, b)), __fsub_rn(x, b));
  acc.h = s;
  acc.l = __fadd_rn(acc.l, __fadd_rn(e, low));
}
// acc += a b
__device__ __forceinline__ void ff_fma(ff &acc, ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  ff_push(acc, p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p))));
}
// a + b, to the last bit the same as b + a: the lanes of a butterfly sum must
// agree, since they rotate their rows by what they compute from it.
__device__ __forceinline__ ff ff_add(ff a, ff b) {
  ff v = ff{a.h, 0.f};
  ff_push(v, b.h, __fadd_rn(a.l, b.l));
  return ff_norm(v);
}
__device__ __forceinline__ ff ff_mul(ff a, ff b) {
  const float p = __fmul_rn(a.h, b.h);
  return ff_norm(ff{p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))});
}
// f (1 + d)^(-1/2) for |d| of the order of single rounding
__device__ __forceinline__ ff ff_corrected(float f, float d) {
  return ff_norm(ff{f, f * (d * fmaf(0.375f, d, -0.5f))});
}
// 1 / sqrt(x), x a normal positive number: the same third-order step as rsqrt64
__device__ __forceinline__ ff ff_rsqrt(ff x) {
  const float r = rsqrtf(x.h), y = __fmul_rn(x.h, r);  // y + yl = x r
  const float yl = fmaf(x.l, r, fmaf(x.h, r, -y));
  return ff_corrected(r, fmaf(yl, r, fmaf(y, r, -1.f)));
}

template <>
struct alignas(16) cplx<ff> {
  ff re, im;
};

// Arithmetic of the working precision S (double or ff).
template <typename S>
struct Work;
template <>
struct Work<double> {
  static constexpr double eps = 1.11e-16, tiny2 = 1e-32;
  static __device__ __forceinline__ double minus(double x) { return -x; }
  static __device__ __forceinline__ double scale(double x, float) { return x; }
  // order of the high words, then (low bits) the lower column first
  static __device__ __forceinline__ int key(double x, int c) {
    const int hi = __double2hiint(x);
    return hi < 0 ? -1 : ((hi & ~127) | (127 - c));
  }
  static constexpr int key_infinite = 0x7ff00000;
  static __device__ __forceinline__ double infinite() { return __longlong_as_double(0x7ff0000000000000ll); }
  static __device__ __forceinline__ double value(double x) { return x; }
  static __device__ __forceinline__ bool finite(double x) { return x <= 1.7e308; }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ double norm(double a) { return a; }
  static __device__ __forceinline__ double of(double x) { return x; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double rsqrt(double x) { return rsqrt64(x); }
  // w += conj(a) b, b -= u w, s += |x|^2
  static __device__ __forceinline__ void dot(cplx<double> &w, cplx<double> a, cplx<double> b) { cfma(w, cconj(a), b); }
  static __device__ __forceinline__ void axpy(cplx<double> &b, cplx<double> u, cplx<double> w) {
    cfma(b, cmake<double>(-u.re, -u.im), w);
  }
  static __device__ __forceinline__ void sq(double &s, cplx<double> x) { s = fma(x.re, x.re, fma(x.im, x.im, s)); }
  static __device__ __forceinline__ double shfl(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
};
template <>
struct Work<float> {
  static __device__ __forceinline__ float add(float a, float b) { return a + b; }
  static __device__ __forceinline__ float norm(float a) { return a; }
  static __device__ __forceinline__ float shfl(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
};
template <>
struct Work<ff> {
  static constexpr float eps = 1.42e-14f, tiny2 = 1e-28f;  // 2^-46
  static __device__ __forceinline__ ff minus(ff x) { return ff_neg(x); }
  static __device__ __forceinline__ ff scale(float x, float sc) { return ff_of(x * sc); }
  static __device__ __forceinline__ int key(ff x, int c) {
    const int b = __float_as_int(x.h);
    return b < 0 ? -1 : ((b & ~127) | (127 - c));
  }
  static constexpr int key_infinite = 0x7f800000;
  static __device__ __forceinline__ ff infinite() { return ff_of(__int_as_float(0x7f800000)); }
  static __device__ __forceinline__ float value(ff x) { return x.h; }
  static __device__ __forceinline__ bool finite(ff x) { return x.h <= 3e38f; }
  static __device__ __forceinline__ ff add(ff a, ff b) { return ff_add(a, b); }
  static __device__ __forceinline__ ff norm(ff a) { return ff_norm(a); }
  static __device__ __forceinline__ ff of(float x) { return ff_of(x); }
  static __device__ __forceinline__ ff mul(ff a, ff b) { return ff_mul(a, b); }
  static __device__ __forceinline__ ff rsqrt(ff x) { return ff_rsqrt(x); }
  static __device__ __forceinline__ void dot(cplx<ff> &w, cplx<ff> a, cplx<ff> b) {
    ff_fma(w.re, a.re, b.re);
    ff_fma(w.re, a.im, b.im);
    ff_fma(w.im, a.re, b.im);
    ff_fma(w.im, ff_neg(a.im), b.re);
  }
  static __device__ __forceinline__ void axpy(cplx<ff> &b, cplx<ff> u, cplx<ff> w) {
    const ff nr = ff_neg(u.re), ni = ff_neg(u.im);
    ff_fma(b.re, nr, w.re);
    ff_fma(b.re, u.im, w.im);
    ff_fma(b.im, nr, w.im);
    ff_fma(b.im, ni, w.re);
    b.re = ff_norm(b.re);
    b.im = ff_norm(b.im);
  }
  static __device__ __forceinline__ void sq(ff &s, cplx<ff> x) {
    ff_fma(s, x.re, x.re);
    ff_fma(s, x.im, x.im);
  }
  static __device__ __forceinline__ ff shfl(ff v, int o) {
    return ff{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)};
  }
};

// Sum over the lanes of a group (from = kGroup / 2) or a warp (from = 16).
template <typename S>
__device__ __forceinline__ S lane_sum(S v, int from) {
  v = Work<S>::norm(v);
#pragma unroll
  for (int o = from; o > 0; o >>= 1) v = Work<S>::add(v, Work<S>::shfl(v, o));
  return v;
}
__device__ __forceinline__ double group_sum(double v) { return lane_sum<double>(v, kGroup / 2); }
__device__ __forceinline__ ff group_sum(ff v) { return lane_sum<ff>(v, kGroup / 2); }
// Both parts of a complex number: at the first level half of the lanes take
// over the real and half the imaginary part, so the sum costs the additions of
// one number.
template <typename S>
__device__ __forceinline__ cplx<S> group_sum(cplx<S> w) {
  const bool upper = (lane_id() & (kGroup / 2)) != 0;
  const S re = Work<S>::norm(w.re), im = Work<S>::norm(w.im);
  S v = Work<S>::add(upper ? im : re, Work<S>::shfl(upper ? re : im, kGroup / 2));
#pragma unroll
  for (int o = kGroup / 4; o > 0; o >>= 1) v = Work<S>::add(v, Work<S>::shfl(v, o));
  const S other = Work<S>::shfl(v, kGroup / 2);
  return cmake<S>(upper ? other : v, upper ? v : other);
}

// Scalars of the Hermitian reflector P = I - v v^dag of a column x with squared
// norm nx2 > 0 and first element al: P x = gamma e_1, gamma = -(al / |al|)
// ||x||, v = (x - gamma e_1) sc with 1 / sc^2 = ||x|| (||x|| + |al|).  Both
// follow from q = 1 / (||x|| |al|): two square roots in a chain instead of
// three.  An |al| below rounding takes the phase 1.
template <typename S>
__device__ __forceinline__ void reflector_scalars(cplx<S> al, S nx2, cplx<S> &gam, S &sc) {
  using K = Work<S>;
  S a2 = K::of(0);
  K::sq(a2, al);
  a2 = K::norm(a2);
  const bool tiny = !(K::value(a2) > K::tiny2 * K::value(nx2));
  if (tiny) {
    al = cmake<S>(K::of(1), K::of(0));
    a2 = K::of(1);
  }
  const S p = K::mul(nx2, a2), q = K::rsqrt(p), t = K::mul(nx2, q);  // t = ||x|| / |al|
  const S mt = K::minus(t);
  gam = cmake<S>(K::mul(al.re, mt), K::mul(al.im, mt));
  sc = K::rsqrt(tiny ? nx2 : K::add(nx2, K::mul(p, q)));
}

// The same for squared norms far from 1, whose products with |al|^2 could leave
// the range of S.
__device__ __forceinline__ void reflector_scaled(cplx<double> al, double nx2, cplx<double> &gam, double &sc) {
  if (nx2 > 1e-130 && nx2 < 1e130) {
    reflector_scalars<double>(al, nx2, gam, sc);
  } else {
    const double r = rsqrt64(nx2);
    reflector_scalars<double>(cscale(al, r), 1.0, gam, sc);
    gam = cscale(gam, nx2 * r);
    sc *= r;
  }
}
// Reflector of the column x[j..m-1] (elements `stride` apart) in the storage
// precision T.  A column of norm up to 1e-30 gets none (sc = 0), one that is not
// finite gets a NaN on the diagonal.  Norm and scalars
// in double, or for float in ff; for float on the column times the power of two
// `down`: single-precision squares of entries near 1e-20 would be denormal, and a
// reflector built from such a norm not unitary.  `unit` makes it P = I - 2 u u^dag
// of a unit u.  One warp.
template <typename T>
struct Reflector {
  cplx<T> gam;  // of the scaled column
  T sc, down, up;
  __device__ __forceinline__ cplx<T> vector(cplx<T> x, bool first) const {
    x = cscale(x, down);
    if (first) x = cmake<T>(x.re - gam.re, x.im - gam.im);
    return sc > T(0) ? cscale(x, sc) : cmake<T>(0, 0);
  }
  __device__ __forceinline__ cplx<T> diagonal() const { return cscale(gam, up); }
};
__device__ __forceinline__ Reflector<double> column_reflector(const cplx<double> *col, int stride, int j, int m,
                                                              bool unit) {
  double s = 0;
  for (int i = j + lane_id(); i < m; i += 32) Work<double>::sq(s, col[i * stride]);
  s = lane_sum<double>(s, 16);
  Reflector<double> h{cmake<double>(0, 0), 0.0, 1.0, 1.0};
  if (!(s <= 1e-60)) reflector_scaled(col[j * stride], s, h.gam, h.sc);  // a NaN goes on into gam
  if (unit) h.sc *= 0.70710678118654752440;
  return h;
}
// Squared norm of a float column scaled by 2^-(ex - 127).  The sum over the warp is
// taken in integers, of steps 2^-20 and 2^-42 (the largest component is in [1, 2),
// so 256 squares give 2^30 of the first), or 2^-17 and 2^-36 for 129 to 1024 rows:
// two integer reductions for five levels of shuffles, and no rounding between.
// Adding a constant with the step as its last place rounds a square to the step,
// and the integer is the difference of the bit patterns.
__device__ __forceinline__ ff column_norm2(const cplx<float> *col, int stride, int j, int m, int &ex) {
  int bits = 0;  // of the largest component: infinity and, above it, NaN among them
  for (int i = j + lane_id(); i < m; i += 32)
    bits = max(bits, max(__float_as_int(fabsf(col[i * stride].re)), __float_as_int(fabsf(col[i * stride].im))));
  bits = __reduce_max_sync(0xffffffffu, bits);
  ex = min(253, max(1, bits >> 23));
  const float down = __int_as_float((254 - ex) << 23);
  if (m > 1024) {
    ff s = ff_of(0.f);
    for (int i = j + lane_id(); i < m; i += 32) {
      const float re = col[i * stride].re * down, im = col[i * stride].im * down;
      ff_fma(s, ff_of(re), ff_of(re));
      ff_fma(s, ff_of(im), ff_of(im));
    }
    return lane_sum<ff>(s, 16);
  }
  const bool tall = m > 128;
  const float c1 = tall ? 0x1.8p6f : 0x1.8p3f, c2 = tall ? 0x1.8p-13f : 0x1.8p-19f;
  const float step1 = tall ? 0x1p-17f : 0x1p-20f, step2 = tall ? 0x1p-36f : 0x1p-42f;
  int hi = 0, lo = 0;
  auto square = [&](float x) {
    const float p = __fmul_rn(x, x), e = fmaf(x, x, -p);
    const float s1 = __fadd_rn(p, c1), r = __fadd_rn(__fsub_rn(p, __fsub_rn(s1, c1)), e);
    hi += __float_as_int(s1) - __float_as_int(c1);
    lo += __float_as_int(__fadd_rn(r, c2)) - __float_as_int(c2);
  };
  for (int i = j + lane_id(); i < m; i += 32) {
    square(col[i * stride].re * down);
    square(col[i * stride].im * down);
  }
  const int th = __reduce_add_sync(0xffffffffu, hi), tl = __reduce_add_sync(0xffffffffu, lo);
  ff s = ff_norm(ff{static_cast<float>(th & ~4095) * step1, static_cast<float>(th & 4095) * step1});
  s.l = fmaf(static_cast<float>(tl), step2, s.l);
  s = ff_norm(s);
  if (bits >= 0x7f800000) s.h = __int_as_float(bits);  // the integers say nothing then
  return s;
}
__device__ __forceinline__ Reflector<float> column_reflector(const cplx<float> *col, int stride, int j, int m,
                                                             bool unit) {
  int ex;
  const ff s = column_norm2(col, stride, j, m, ex);
  Reflector<float> h{cmake<float>(0.f, 0.f), 0.f, __int_as_float((254 - ex) << 23), __int_as_float(ex << 23)};
  if (ex > 30 || sqrtf(s.h) * h.up > 1e-30f) {
    cplx<ff> g;
    ff c;
    const cplx<float> al = cscale(col[j * stride], h.down);
    reflector_scalars<ff>(cmake<ff>(ff_of(al.re), ff_of(al.im)), s, g, c);
    h.gam = cmake<float>(g.re.h, g.im.h);
    h.sc = unit ? ff_mul(c, ff{0.70710677f, 1.2101617e-8f}).h : c.h;
  }
  return h;
}

// 1 / x of a normal x: the hardware's approximation r and, with e = 1 - x r, the
// geometric series r (1 + e + ...) to e^2 for double, to e for the float of a pair;
// within one unit in the last place.
__device__ __forceinline__ double reciprocal(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r * e, 1.0 + e, r);
}
__device__ __forceinline__ float reciprocal(ff x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x.h));
  return fmaf(r, fmaf(-x.l, r, fmaf(-x.h, r, 1.f)), r);
}

// Reflector j of a column x (rows j.. m-1) without writing its vector: P = I -
// beta v v^dag with v = (v0, x_{j+1}, ...), P x = gam e_1, gam = -(x_j / |x_j|)
// ||x||, v0 = x_j - gam, beta = 1 / (||x|| (||x|| + |x_j|)).  The rows below j are v
// as they stand, so v^dag b over them needs no scalar of the reflector, and beta
// needs a reciprocal where a normalised v needs a second root.  A column of norm up
// to 1e-30 gets beta = 0.  A column so far from 1 that beta leaves the range is
// scaled by a power of two (moved).  Scalars in double, or for float in ff, of the
// column times a power of two.  One warp.
template <typename T>
struct ColumnHead {
  cplx<T> v0, gam;
  T beta, moved;
};
template <typename S>
__device__ __forceinline__ void head_scalars(cplx<S> al, S nx2, cplx<S> &v0, cplx<S> &gam, S &h) {
  using K = Work<S>;
  S a2 = K::of(0);
  K::sq(a2, al);
  a2 = K::norm(a2);
  const bool tiny = !(K::value(a2) > K::tiny2 * K::value(nx2));  // takes the phase 1
  const cplx<S> ph = tiny ? cmake<S>(K::of(1), K::of(0)) : al;
  const S p = tiny ? nx2 : K::mul(nx2, a2), q = K::rsqrt(p), t = K::minus(K::mul(nx2, q));
  gam = cmake<S>(K::mul(ph.re, t), K::mul(ph.im, t));
  v0 = cmake<S>(K::add(al.re, K::minus(gam.re)), K::add(al.im, K::minus(gam.im)));
  h = tiny ? nx2 : K::add(nx2, K::mul(p, q));
}
__device__ __forceinline__ void column_head(cplx<double> *col, int j, int m, ColumnHead<double> *out) {
  double sr = 0, si = 0;
  for (int i = j + lane_id(); i < m; i += 32) {
    sr = fma(col[i].re, col[i].re, sr);
    si = fma(col[i].im, col[i].im, si);
  }
  double s = sr + si;
  for (int o = 16; o > 0; o >>= 1)  // lanes past the column hold zero
    if (o < m - j) s += __shfl_xor_sync(0xffffffffu, s, o);
  s = __shfl_sync(0xffffffffu, s, 0);
  cplx<double> al = col[j];
  ColumnHead<double> r{cmake<double>(0, 0), cmake<double>(0, 0), 0.0, 0.0};
  if (!(s <= 1e-60)) {
    double up = 1.0;
    if (s > 1e130) {
      const int ex = min(2045, max(1, (__double2hiint(s) >> 21) + 512));  // half the exponent of s, biased
      up = __hiloint2double(ex << 20, 0);
      const double down = __hiloint2double((2046 - ex) << 20, 0);
      for (int i = j + 1 + lane_id(); i < m; i += 32) col[i] = cscale(col[i], down);
      al = cscale(al, down);
      s = s * down * down;
      r.moved = 1.0;
    }
    double h;
    head_scalars<double>(al, s, r.v0, r.gam, h);
    r.gam = cscale(r.gam, up);
    r.beta = reciprocal(h);
  }
  if (lane_id() == 0) *out = r;
}
__device__ __forceinline__ void column_head(cplx<float> *col, int j, int m, ColumnHead<float> *out) {
  int ex;
  const ff s = column_norm2(col, 1, j, m, ex);
  const float down = __int_as_float((254 - ex) << 23), up = __int_as_float(ex << 23);
  ColumnHead<float> r{cmake<float>(0.f, 0.f), cmake<float>(0.f, 0.f), 0.f, 0.f};
  if (ex > 30 || sqrtf(s.h) * up > 1e-30f) {  // 2^-97 is above 1e-30
    const bool far = ex < 97 || ex > 157;  // entries up to 2^-30 or from 2^31
    const cplx<float> al = cscale(col[j], down);
    cplx<ff> v0, gam;
    ff h;
    head_scalars<ff>(cmake<ff>(ff_of(al.re), ff_of(al.im)), s, v0, gam, h);
    const float vs = far ? 1.f : up, bs = far ? 1.f : down;
    r.v0 = cmake<float>(v0.re.h * vs, v0.im.h * vs);
    r.gam = cmake<float>(gam.re.h * up, gam.im.h * up);
    r.beta = reciprocal(h) * bs * bs;
    r.moved = far ? 1.f : 0.f;
    if (far)
      for (int i = j + 1 + lane_id(); i < m; i += 32) col[i] = cscale(col[i], down);
  }
  if (lane_id() == 0) *out = r;
}

// The same for a column whose squared norm is known, in the working precision: v0,
// gam and beta to out[0], out[1] and out[2].re.  One warp.
__device__ __forceinline__ void head_scaled(cplx<double> al, double nx2, cplx<double> *out) {
  cplx<double> v0, gam;
  double h, f = 1.0, g = 1.0;
  if (!(nx2 > 1e-130 && nx2 < 1e130)) {
    const int ex = min(1535, max(512, (__double2hiint(nx2) >> 21) + 512));  // half the exponent of nx2, biased
    f = __hiloint2double((2046 - ex) << 20, 0);
    g = __hiloint2double(ex << 20, 0);
  }
  head_scalars<double>(cscale(al, f), nx2 * f * f, v0, gam, h);
  if (lane_id() == 0) {
    out[0] = cscale(v0, g);
    out[1] = cscale(gam, g);
    out[2].re = reciprocal(h) * f * f;
  }
}
__device__ __forceinline__ void head_scaled(cplx<ff> al, ff nx2, cplx<ff> *out) {
  const int e = (__float_as_int(nx2.h) >> 24) - 63;  // nx2 in [2^(2 e - 1), 2^(2 e + 1))
  const float f = __int_as_float((127 - e) << 23), g = __int_as_float((127 + e) << 23);
  auto times = [](ff x, float y) { return ff{x.h * y, x.l * y}; };  // by a power of two
  cplx<ff> v0, gam;
  ff h;
  head_scalars<ff>(cmake<ff>(times(al.re, f), times(al.im, f)), times(times(nx2, f), f), v0, gam, h);
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(h.h));
  const float e1 = fmaf(-h.l, r, fmaf(-h.h, r, 1.f));  // the same series, to e^2, as a pair
  const ff beta = ff_norm(ff{r, r * fmaf(e1, e1, e1)});
  if (lane_id() == 0) {
    out[0] = cmake<ff>(times(v0.re, g), times(v0.im, g));
    out[1] = cmake<ff>(times(gam.re, g), times(gam.im, g));
    out[2].re = times(times(beta, f), f);
  }
}

// v^dag b over the rows below j of a group's lanes: two accumulators a part, so
// that a row costs one dependent operation
template <typename T>
__device__ __forceinline__ cplx<T> dot_below(const cplx<T> *x, const cplx<T> *b, int i0, int m) {
  T r0 = 0, r1 = 0, q0 = 0, q1 = 0;
#pragma unroll 4
  for (int i = i0; i < m; i += kGroup) {
    const cplx<T> u = x[i], v = b[i];
    r0 = fma(u.re, v.re, r0);
    r1 = fma(u.im, v.im, r1);
    q0 = fma(u.re, v.im, q0);
    q1 = fma(-u.im, v.re, q1);
  }
  return cmake<T>(r0 + r1, q0 + q1);
}

// Householder QR in shared memory.  A is m x n: row-major with leading
// dimension lda (conj_t false), or given as its conjugate transpose, an n x m
// row-major array with leading dimension lda (conj_t true).  R (min(m, n) rows,
// zero below the diagonal, then zero rows up to r_rows) goes to Rout, row-major
// with leading dimension n; Rout may be A.  With Qout, the explicit Q (m x
// min(m, n)) goes there row-major, or with conj_t its conjugate transpose
// (min(m, n) x m); Qout may be A.  buf holds qr_small_elems elements: the columns
// (which keep the reflectors' rows below the diagonal), the reflectors' heads,
// then Q.  CTA-wide.
//
// The vectors are not normalised, so v^dag b is a product of two columns' sizes:
// entries have to stay below 2^60 in complex64 and 2^300 in complex128, as those of
// a state do.
//
// What bounds a column is a chain: its norm, a root and a reciprocal (about 600
// cycles for ff, 1400 for double, whose operations take 64 each), then the
// update.  One warp that owns no column runs the chain while the others form
// v^dag b of theirs; between, two barriers of the warps involved.
// Against a chain that ran from the update of the next column to its normalised
// reflector, before any v^dag b: a d = 5 round at theta = 1e-3 88.4 -> 86.8 ms, a
// 40 x 20 complex128 R factor 82 -> 69 us, d = 5 pairs in complex128 243 -> 233 ms.
//
// The blocked routine (qr_r_inplace) keeps its trailing columns in global memory.
__host__ __device__ __forceinline__ int64_t qr_small_elems(int m, int n, bool with_q) {
  const int64_t ld = m | 1, steps = m < n ? m : n;
  return ld * (n + (with_q ? steps : 0)) + 3 * steps;
}

template <typename T>
static __device__ __noinline__ void qr_small(int m, int n, const cplx<T> *A, int lda, bool conj_t, cplx<T> *Rout,
                                             int r_rows, cplx<T> *Qout, cplx<T> *buf_) {
  const int ld = m | 1, steps = min(m, n);
  cplx<T> *Bm = in_smem<cplx<T>>(buf_);
  static_assert(sizeof(ColumnHead<T>) == 3 * sizeof(cplx<T>), "qr_small_elems");
  ColumnHead<T> *head = in_smem<ColumnHead<T>>(Bm + n * ld);
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
  // the last warp finds the scalars; it owns columns only where all warps have to
  const bool spare = team_threads(n) < kThreads;
  const int nthr = team_threads(n) + (spare ? 32 : 0);
  const int gl = lane_id() & (kGroup - 1), g = tid() / kGroup, groups = nthr / kGroup - (spare ? 4 : 0);
  if (tid() < nthr) {
    const bool scalars = tid() >= nthr - 32, owns = g < groups;
    for (int j = 0; j < steps; ++j) {
      const cplx<T> *x = Bm + j * ld;
      // a lane keeps its rows, i = gl (mod 8): its first one below row j, and from it
      const int i0 = j + 1 + ((gl - j - 1) & (kGroup - 1)), ij = j + ((gl - j) & (kGroup - 1));
      // columns j + 1 .. n - 1 in turn, column c to group c % groups
      int c = j + 1 + (g - (j + 1) % groups + groups) % groups;
      cplx<T> w = cmake<T>(0, 0);
      if (scalars) {
        column_head(Bm + j * ld, j, m, head + j);
      }
      if (owns && j + 1 < n) {
        if (c < n) w = dot_below(x, Bm + c * ld, i0, m);
        w = group_sum(w);
      }
      team_sync(nthr);
      if (owns) {
        const ColumnHead<T> h = head[j];
        for (int k = 0; k * groups < n - j - 1; ++k, c += groups) {  // warp-uniform trip count
          cplx<T> *b = Bm + min(c, n - 1) * ld;
          if (k > 0 || h.moved != T(0)) {
            w = cmake<T>(0, 0);
            if (c < n) w = dot_below(x, b, i0, m);
            w = group_sum(w);
          }
          const cplx<T> bj = b[j];
          __syncwarp();
          if (c < n) {
            cfma(w, cconj(h.v0), bj);
            w = cscale(w, -h.beta);
#pragma unroll 4
            for (int i = ij; i < m; i += kGroup) {
              cplx<T> y = b[i];
              cfma(y, i == j ? h.v0 : x[i], w);
              b[i] = y;
            }
          }
        }
      }
      team_sync(nthr);
    }
  }
  __syncthreads();
  for (int e = tid(); e < r_rows * n; e += kThreads) {
    const int i = e / n, c = e % n;
    Rout[e] = i < steps && c >= i ? (c == i ? head[i].gam : Bm[c * ld + i]) : cmake<T>(0, 0);
  }
  if (Qout == nullptr) {
    __syncthreads();
    return;
  }
  // Q e_c = P_0 ... P_c e_c (a reflector below row c leaves e_c alone)
  cplx<T> *Qm = reinterpret_cast<cplx<T> *>(head + steps);
  for (int c = tid() / kGroup; (c & ~3) < steps; c += kGroups) {
    const int top = min(steps - 1, (c & ~3) + 3);  // largest column of the warp
    cplx<T> *q = Qm + min(c, steps - 1) * ld;
    const bool col = c < steps;
    if (col)
      for (int i = gl; i < m; i += kGroup) q[i] = cmake<T>(i == c ? T(1) : T(0), 0);
    __syncwarp();
    for (int j = top; j >= 0; --j) {
      const cplx<T> *x = Bm + j * ld;
      const int i0 = j + 1 + ((gl - j - 1) & (kGroup - 1));
      const bool on = col && j <= c;
      const ColumnHead<T> h = head[j];
      cplx<T> w = cmake<T>(0, 0);
      if (on) {
        w = dot_below(x, q, i0, m);
        if (gl == (j & (kGroup - 1))) cfma(w, cconj(h.v0), q[j]);
      }
      w = group_sum(w);
      if (on) {
        w = cscale(w, -h.beta);
#pragma unroll 4
        for (int i = i0; i < m; i += kGroup) {
          cplx<T> y = q[i];
          cfma(y, x[i], w);
          q[i] = y;
        }
        if (gl == (j & (kGroup - 1))) {
          cplx<T> y = q[j];
          cfma(y, h.v0, w);
          q[j] = y;
        }
      }
    }
  }
  __syncthreads();
  for (int e = tid(); e < m * steps; e += kThreads) {
    if (!conj_t) {
      const int i = e / steps, c = e % steps;
      Qout[e] = Qm[c * ld + i];
    } else {
      const int c = e / m, i = e % m;
      Qout[e] = cconj(Qm[c * ld + i]);
    }
  }
  __syncthreads();
}

// The rotation of a pair of rows with squared norms al, be and inner product
// g: x <- cs x - sn uc y, y <- sn x + cs uc y makes them orthogonal.  Its angle
// is found in single precision from numbers scaled by a power of two; cosine,
// sine and the phase uc = conj(g / |g|) are then brought to the working
// precision by a third-order correction, so the rotation is unitary to rounding
// and only its angle is approximate (which costs no sweep: an angle good to a few
// 1e-7 leaves that much of the product).  So the angle and the test whether there
// is one to rotate by use the hardware's approximate reciprocal and root.  tg: what |x|^2 loses and |y|^2 gains;
// reach: |tan| sqrt(max / min) of the norms, at least 0.8 of the rows' cosine.
template <typename S>
struct Rotation {
  S cs, sn, tg;
  cplx<S> uc;
  float reach;
};

__device__ __forceinline__ float fast_reciprocal(float x) {
  float r;
  asm("rcp.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float fast_root(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void rotation_angle(float diff, float gr, float gi, float &t, float &ur, float &ui,
                                               float &absg) {
  const float mx = fmaxf(fmaxf(fabsf(gr), fabsf(gi)), 1e-37f), imx = fast_reciprocal(mx);
  const float a = gr * imx, b = gi * imx, n2 = a * a + b * b, rn = rsqrtf(n2);
  absg = mx * (n2 * rn);
  const float zeta = 0.5f * diff * fast_reciprocal(absg), az = fabsf(zeta);
  t = az > 1e10f ? 0.5f * fast_reciprocal(az) : fast_reciprocal(az + fast_root(1.f + az * az));
  if (zeta < 0.f) t = -t;
  ur = a * rn;
  ui = -b * rn;
}

__device__ __forceinline__ bool make_rotation(double al, double be, cplx<double> g, float tol, Rotation<double> &r) {
  // the larger norm is scaled to [1, 2) and the rest seen in single precision: a
  // double-precision comparison of the squares takes five operations of 64 cycles
  const int ex = min(2045, max(1, max(__double2hiint(al), __double2hiint(be)) >> 20));
  const double sc = __hiloint2double((2046 - ex) << 20, 0);
  const float af = static_cast<float>(al * sc), bf = static_cast<float>(be * sc);
  const float gr = static_cast<float>(g.re * sc), gi = static_cast<float>(g.im * sc);
  const float root = fast_root(af) * fast_root(bf), lim = tol * root;
  if (!(fmaxf(fabsf(gr), fabsf(gi)) > 0.70711f * lim)) return false;  // max(|re|, |im|) >= |g| / sqrt(2)
  float tf, urf, uif, absg;
  rotation_angle(static_cast<float>((be - al) * sc), gr, gi, tf, urf, uif, absg);
  if (!(absg > lim)) return false;
  const double t = static_cast<double>(tf), w = fma(t, t, 1.0);
  const double c0 = static_cast<double>(rsqrtf(fmaf(tf, tf, 1.f)));
  double d = fma(-w * c0, c0, 1.0);
  r.cs = fma(c0 * d, fma(0.375, d, 0.5), c0);
  r.sn = t * r.cs;
  const double ur = static_cast<double>(urf), ui = static_cast<double>(uif);
  d = fma(-ur, ur, fma(-ui, ui, 1.0));
  d = fma(d, fma(0.375, d, 0.5), 1.0);
  r.uc = cmake<double>(ur * d, ui * d);
  r.tg = static_cast<double>(tf * absg) * __hiloint2double(ex << 20, 0);
  r.reach = fabsf(tf) * fmaxf(af, bf) * fast_reciprocal(root);
  return true;
}
__device__ __forceinline__ bool make_rotation(ff al, ff be, cplx<ff> g, float tol, Rotation<ff> &r) {
  const float gr = g.re.h, gi = g.im.h;
  const float lim = tol * fast_root(al.h) * fast_root(be.h);
  if (!(fmaxf(fabsf(gr), fabsf(gi)) > 0.70711f * lim)) return false;  // max(|re|, |im|) >= |g| / sqrt(2)
  float tf, ur, ui, absg;
  rotation_angle(ff_add(be, ff_neg(al)).h, gr, gi, tf, ur, ui, absg);
  if (!(absg > lim)) return false;
  const ff t = ff_of(tf);
  ff w = ff_of(1.f);
  ff_fma(w, t, t);
  r.cs = ff_rsqrt(ff_norm(w));
  r.sn = ff_mul(t, r.cs);
  ff d = ff_of(-1.f);
  ff_fma(d, ff_of(ur), ff_of(ur));
  ff_fma(d, ff_of(ui), ff_of(ui));
  r.uc = cmake<ff>(ff_corrected(ur, d.h + d.l), ff_corrected(ui, d.h + d.l));
  r.tg = ff_of(tf * absg);
  r.reach = fabsf(tf) * fmaxf(al.h, be.h) * tol * fast_reciprocal(lim);
  return true;
}

__device__ __forceinline__ void rotate_pair(cplx<double> &x, cplx<double> &y, const Rotation<double> &r) {
  const cplx<double> a = x, b = cmul(r.uc, y);
  x = cmake<double>(fma(r.cs, a.re, -r.sn * b.re), fma(r.cs, a.im, -r.sn * b.im));
  y = cmake<double>(fma(r.sn, a.re, r.cs * b.re), fma(r.sn, a.im, r.cs * b.im));
}
// a b + c d
__device__ __forceinline__ ff ff_two(ff a, ff b, ff c, ff d) {
  const float p = __fmul_rn(a.h, b.h);
  ff v = ff{p, fmaf(a.l, b.h, fmaf(a.h, b.l, fmaf(a.h, b.h, -p)))};
  ff_fma(v, c, d);
  return ff_norm(v);
}
__device__ __forceinline__ void rotate_pair(cplx<ff> &x, cplx<ff> &y, const Rotation<ff> &r) {
  const cplx<ff> a = x;
  const cplx<ff> b = cmake<ff>(ff_two(r.uc.re, y.re, ff_neg(r.uc.im), y.im), ff_two(r.uc.re, y.im, r.uc.im, y.re));
  const ff ns = ff_neg(r.sn);
  x = cmake<ff>(ff_two(r.cs, a.re, ns, b.re), ff_two(r.cs, a.im, ns, b.im));
  y = cmake<ff>(ff_two(r.sn, a.re, r.cs, b.re), ff_two(r.sn, a.im, r.cs, b.im));
}

// Keep count at one bond from its eigenvalues lam (>= 0) in the decreasing order
// perm, by one warp.  The cutoff is compared in squares, lam_i > cutoff^2 lam_1:
// square roots (of double, by one thread) were most of the 11,000 cycles the
// keep decision of a bond took.
template <typename T>
static __device__ int keep_count(const T *lam, const int *perm, int n, int cap, double cutoff, double delta) {
  auto at = [&](int i) { return static_cast<double>(lam[perm[i]]); };
  auto above = [&](int m, double thr2) {
    int k = 0;
    for (int i = 0; i < m; i += 32)
      k += __popc(__ballot_sync(0xffffffffu, i + lane_id() < m && at(min(i + lane_id(), m - 1)) > thr2));
    return k;
  };
  const double l1 = at(0);
  if (!(l1 > 0.0)) return 1;
  int k;
  if constexpr (sizeof(T) == 4) {  // a float is above a bound if it is above the float below that
    const float thr = __double2float_rd(cutoff * cutoff * l1);
    k = 0;
    for (int i = 0; i < n; i += 32)
      k += __popc(__ballot_sync(0xffffffffu, i + lane_id() < n && lam[perm[min(i + lane_id(), n - 1)]] > thr));
    k = max(1, k);
  } else {
    k = max(1, above(n, cutoff * cutoff * l1));
  }
  if (k > cap) {
    const double c = at(cap);  // (sqrt(c) + delta sqrt(l1))^2, and c itself at delta = 0
    k = max(1, above(cap, c + delta * (2.0 * sqrt(c * l1) + delta * l1)));
  }
  return k;
}

// Discarded over total weight of a bond, by one warp (lane 0's value counts);
// left: the lane's share of a weight that is not in lam, discarded too.
static __device__ __forceinline__ double discarded_weight(const double *lam, const int *perm, int n, int keep,
                                                          double left = 0) {
  double tot = left, drop = left;
  for (int i = lane_id(); i < n; i += 32) {
    const double l = lam[perm[i]];
    tot += l;
    if (i >= keep) drop += l;
  }
  tot = warp_sum(tot);
  drop = warp_sum(drop);
  return tot > 0 ? drop / tot : 0.0;
}
static __device__ __forceinline__ double discarded_weight(const float *lam, const int *perm, int n, int keep,
                                                          float left = 0) {
  ff tot = ff_of(left), drop = tot;
  for (int i = lane_id(); i < n; i += 32) {
    const float l = lam[perm[i]];
    ff_push(tot, l, 0.f);
    if (i >= keep) ff_push(drop, l, 0.f);
  }
  tot = lane_sum<ff>(tot, 16);
  drop = lane_sum<ff>(drop, 16);
  if (!(tot.h > 0.f)) return 0.0;
  const float q = drop.h / tot.h;
  ff_fma(drop, ff_of(-q), tot);  // the remainder: a second quotient digit of single precision
  return static_cast<double>(q) + static_cast<double>((drop.h + drop.l) / tot.h);
}

// What the truncation wants of a bond's SVD: the order of its values, how many are
// kept (of at most kmax; also the result of svd_small) and the kept vectors.
template <typename T>
struct Truncation {
  int *perm;      // decreasing order of lam (shared memory)
  int kmax;
  double delta;
  int *fail, *keep;
  double *discarded;  // the discarded over the total weight is added
  cplx<T> *vs, *site;  // n x keep vectors and, in complex64, the keep x n site of their conjugates
};

// SVD of a bond in shared memory, in double precision (T = double) or in
// pairs of floats (T = float): Householder QR with column pivoting, then
// one-sided (Hestenes) Jacobi on the rows of R, the preconditioning of Drmac
// and Veselic (SIAM J. Matrix Anal. Appl. 29, 2008).  A (m x n, row-major,
// leading dimension n) = Q R, R in the original column order; rotating the rows
// of R until they are orthogonal gives the rows sigma_i v_i^dag, so no rotation
// is accumulated.  lam[i] = sigma_i^2 (unsorted, zero beyond the numerical rank,
// which is returned) and column i of V (n x n, column-major; columns beyond the
// rank are not written, except column 0 of a zero matrix) = v_i.  A row of R whose
// norm falls below rounding counts as zero: it was not rotated any more, so it
// gives no vector.  Values that are not finite give lam = NaN.
//
// Against Jacobi on A's columns with accumulated V this takes about half the
// sweeps and a quarter of the rotations on the matrices of a d = 3 and a d = 5
// run, and rotates one matrix instead of two.
//
// Pairs of floats against double, on the complex64 path whose input and output
// are single precision: 32 x 32 bonds of a d = 5 round take 259 us against 960
// us, 52 x 52 ones of an X-memory 0.84 ms against 3.1 ms, with the same errors
// of the singular values, vectors and truncated matrix.
//
// cutoff > 0 (the truncation's): the QR stops once the norm of all that is left
// is at most d sigma_1, d = min(cutoff / 16, sqrt(eps_T cutoff)) with eps_T the
// rounding of T; what is left counts as discarded weight and has no vector, whatever
// the cutoff.  A value below cutoff sigma_1 is dropped by the caller, and
// leaving such a remainder out turns a kept vector of value s by at most (d
// sigma_1 / s)^2, that is the decomposed matrix by d^2 sigma_1 / cutoff <= eps_T
// sigma_1.  In complex64 the remainder is the rounding noise of A, about a third
// of the rows of a bond, and the most expensive ones.  (Keeping them but not
// rotating them against each other was slower: it leaves the sweeps converging
// linearly.)
//
// With tr (the truncation's) V is not written: values are sorted, counted and the
// kept vectors stored from shared memory, without a pass through V and back (with
// the shorter sums of column_norm2 and integer flop counts: a d = 5 round at theta
// = 1e-3 86.4 -> 79.3 ms, d = 7 151.7 -> 138.1 ms).
//
// buf: n (m | 1) 16-byte complex numbers in shared memory, or (SM false) n m of
// them in global memory, for the few bonds that are too large for a CTA that has
// half of an SM: the same arithmetic, so a result does not depend on where the
// matrix was; u: 3 of them; nr: 2 kSmallSvdCols
// doubles (both shared memory; lam too, with tr); n <=
// kSmallSvdCols.  CTA-wide.
template <typename T, bool SM>
static __device__ __noinline__ int svd_small(int m, int n, const cplx<T> *A, cplx<T> *V, T *lam, double cutoff_,
                                             void *buf_, void *u_, void *nr_, const Truncation<T> *tr = nullptr) {
  using S = std::conditional_t<sizeof(T) == 8, double, ff>;
  using K = Work<S>;
  using R = decltype(K::value(S()));  // double or float
  const int ld = SM ? m | 1 : m, steps = min(m, n);
  cplx<S> *Bm, *u = in_smem<cplx<S>>(u_);
  if constexpr (SM) Bm = in_smem<cplx<S>>(buf_);
  else Bm = static_cast<cplx<S> *>(buf_);
  S *nr = in_smem<S>(nr_), *rows = nr + kSmallSvdCols;  // squared norms of the columns and of R's rows
  const int gl = lane_id() & (kGroup - 1), g = tid() / kGroup;
  float down = 1.f, up = 1.f;  // ff: the matrix scaled by a power of two to entries up to 1
  if constexpr (sizeof(T) == 4) {
    int *top = reinterpret_cast<int *>(u);
    if (tid() == 0) *top = 0;
    __syncthreads();
    int bits = 0;
    for (int e = tid(); e < m * n; e += kThreads)
      bits = max(bits, max(__float_as_int(fabsf(A[e].re)), __float_as_int(fabsf(A[e].im))));
    bits = __reduce_max_sync(0xffffffffu, bits);
    if (lane_id() == 0) atomicMax(top, bits);
    __syncthreads();
    const int ex = min(253, max(1, *top >> 23));
    down = __int_as_float((254 - ex) << 23);
    up = __int_as_float(ex << 23);
    __syncthreads();
  }
  for (int e = tid(); e < m * n; e += kThreads) {
    const int i = e / n, c = e % n;
    const cplx<T> x = A[e];
    Bm[c * ld + i] = cmake<S>(K::scale(x.re, down), K::scale(x.im, down));
  }
  __syncthreads();
  // largest of k numbers >= 0 (or -1), column in the low bits; every warp finds
  // it by itself.  Of equal columns the first is the pivot, and of equal values the
  // first row's is kept: where a cap cuts a cluster of orthogonal columns of equal
  // norm, the branch that survives is the first one, which is the branch that a
  // gradient's states share (the last one has no overlap with them).
  auto top_key = [&](int k) {
    int key = -1;
    for (int c = lane_id(); c < k; c += 32) key = max(key, K::key(nr[c], c));
    return __reduce_max_sync(0xffffffffu, key);
  };
  const R cutoff = static_cast<R>(cutoff_), eps_t = sizeof(T) == 8 ? R(1.11e-16) : R(5.96e-8);
  int rank = 0;
  R neg = 0;    // squared norm of a negligible row
  R rest = 0;   // squared norm of the remainder that may be left out
  R left = 0;   // bound on the squared norm of the remainder that was left out
  bool finite = true;
  {
    const bool spare = team_threads(n) < kThreads;
    const int nthr = team_threads(n) + (spare ? 32 : 0), groups = nthr / kGroup - (spare ? 4 : 0);
    const bool scalars = tid() >= nthr - 32, owns = g < groups;
    int last = -1;  // the pivot column of the step before, and its diagonal element
    cplx<S> gam = cmake<S>(K::of(0), K::of(0));
    auto finish = [&](int c, int i0) {
      for (int i = i0 + lane_id(); i < m; i += 32) Bm[c * ld + i] = i == i0 ? gam : cmake<S>(K::of(0), K::of(0));
    };
    if (tid() < nthr) {
      for (int c = g; (c & ~3) < n; c += nthr / kGroup) {
        S s = K::of(0);
        if (c < n)
          for (int i = gl; i < m; i += kGroup) K::sq(s, Bm[c * ld + i]);
        s = group_sum(s);
        if (gl == 0 && c < n) nr[c] = K::finite(s) ? s : K::infinite();
      }
    }
    __syncthreads();
    const int k0 = top_key(n);
    finite = k0 < K::key_infinite;
    const R top = K::value(nr[127 - (k0 & 127)]);
    neg = K::eps * K::eps * top;
    rest = min(cutoff * cutoff / 256, eps_t * cutoff) * top;
    __syncthreads();
    if (tid() < nthr && finite) {
      for (int j = 0; j < steps; ++j) {
        const int key = top_key(n);
        const int p = 127 - (key & 127);
        const S nx2 = key < 0 ? K::of(0) : nr[p];
        left = K::value(nx2) * (n - j);
        if (!(K::value(nx2) > neg) || left <= rest) break;  // what is left is dropped or below rounding
        left = 0;
        // as in qr_small: v^dag b below row j while one warp finds the scalars
        const cplx<S> *x = Bm + p * ld;
        const int i0 = j + ((gl - j) & (kGroup - 1));  // a lane keeps its rows: i = gl (mod 8)
        auto raw = [&](int c, bool on) {
          cplx<S> w = cmake<S>(K::of(0), K::of(0));
          if (on)
#pragma unroll 4
            for (int i = i0; i < m; i += kGroup)
              if (i > j) K::dot(w, x[i], Bm[c * ld + i]);
          return group_sum(w);
        };
        auto open = [&](int c) { return c < n && c != p && K::value(nr[min(c, n - 1)]) >= 0; };
        cplx<S> w = cmake<S>(K::of(0), K::of(0));
        if (scalars) {
          head_scaled(x[j], nx2, u);
          if (last >= 0) finish(last, j - 1);
        }
        if (owns) w = raw(g, open(g));
        team_sync(nthr);
        if (owns) {
          const cplx<S> v0 = u[0];
          const S beta = u[2].re;
          for (int c = g; (c & ~3) < n; c += groups) {
            const bool on = open(c);
            if (__any_sync(0xffffffffu, on)) {
              cplx<S> *b = Bm + min(c, n - 1) * ld;
              if (c != g) w = raw(c, on);
              S s = K::of(0);
              if (on) {
                K::dot(w, v0, b[j]);
                w = cmake<S>(K::mul(K::norm(w.re), beta), K::mul(K::norm(w.im), beta));
              }
              __syncwarp();
              if (on) {
#pragma unroll 4
                for (int i = i0; i < m; i += kGroup) {
                  cplx<S> y = b[i];
                  K::axpy(y, i == j ? v0 : x[i], w);
                  b[i] = y;
                  if (i > j) K::sq(s, y);
                }
              }
              s = group_sum(s);
              if (gl == 0 && on) nr[c] = s;
            }
            __syncwarp();
            if (gl == 0 && c == p) nr[c] = K::of(-1);
          }
        }
        last = p;
        gam = u[1];
        team_sync(nthr);
        rank = j + 1;
      }
      if (scalars && last >= 0) finish(last, rank - 1);
    }
  }
  // the rank is known to the team's threads
  if (tid() == 0) {
    reinterpret_cast<int *>(u)[0] = rank;
    reinterpret_cast<R *>(u)[2] = left;
  }
  __syncthreads();
  rank = reinterpret_cast<int *>(u)[0];
  left = reinterpret_cast<R *>(u)[2];
  __syncthreads();

  // rows of R: row i at Bm[c ld + i], ld odd, so 8 lanes over c meet no bank twice
  const int kk = rank + (rank & 1), half = kk / 2;
  const int nthr = team_threads(max(1, half));
  const R tol = R(4) * K::eps * sqrt(static_cast<R>(n));
  // A sweep whose rotations all stayed within `near` is the last one, without a
  // sweep that only finds nothing left.  A pair made orthogonal is disturbed by
  // the sweep's later rotations of p or q with another row r, each by |tan_pr|
  // <x_r, x_q>: relative to |x_p| |x_q| that is reach_pr times the cosine of (r,
  // q), so at most about reach^2 / 0.8, and there are less than 2 rank of them.
  // near leaves cosines of tol in double, and of 1e-11 in pairs of floats, whose
  // vectors are rounded to float.  Without the last sweep a d = 5 round at theta =
  // 0.05 takes 169 ms instead of 174, at 1e-3 88.5 instead of 92.
  const float near = sqrtf((sizeof(T) == 8 ? static_cast<float>(tol) : 1e-11f) / (2.5f * static_cast<float>(kk)));
  auto norms = [&]() {
    for (int i = g; (i & ~3) < kk; i += nthr / kGroup) {
      S s = K::of(0);
      if (i < rank)
        for (int c = gl; c < n; c += kGroup) K::sq(s, Bm[c * ld + i]);
      s = group_sum(s);
      if (gl == 0 && i < rank) rows[i] = s;
    }
  };
  if (tid() < nthr && finite) {
    for (int sweep = 0; sweep < kMaxSweepsD && rank > 1; ++sweep) {
      norms();
      team_sync(nthr);
      bool again = false;
      for (int round = 0; round < kk - 1; ++round) {
        for (int pi = g; (pi & ~3) < half; pi += nthr / kGroup) {
          int p, q;
          if (pi == 0) { p = kk - 1; q = round; }
          else { p = round + pi; q = round - pi; if (p >= kk - 1) p -= kk - 1; if (q < 0) q += kk - 1; }
          if (p > q) { const int t = p; p = q; q = t; }
          bool on = pi < half && q < rank;
          if (!on) p = q = 0;
          const S al = rows[p], be = rows[q];
          const R av = K::value(al), bv = K::value(be);
          on = on && av > neg && bv > neg;
          if (!__any_sync(0xffffffffu, on)) continue;
          cplx<S> dot = cmake<S>(K::of(0), K::of(0));
          if (on)
#pragma unroll 4
            for (int c = gl; c < n; c += kGroup) K::dot(dot, Bm[c * ld + p], Bm[c * ld + q]);
          dot = group_sum(dot);
          Rotation<S> rot;
          if (on && make_rotation(al, be, dot, static_cast<float>(tol), rot)) {
            again |= rot.reach > near;
#pragma unroll 2
            for (int c = gl; c < n; c += kGroup) {
              cplx<S> x = Bm[c * ld + p], y = Bm[c * ld + q];
              rotate_pair(x, y, rot);
              Bm[c * ld + p] = x;
              Bm[c * ld + q] = y;
            }
            if (gl == 0) {
              const S a1 = K::add(al, K::minus(rot.tg)), b1 = K::add(be, rot.tg);
              rows[p] = K::value(a1) > 0 ? a1 : K::of(0);
              rows[q] = K::value(b1) > 0 ? b1 : K::of(0);
            }
          }
        }
        team_sync(nthr);
      }
      if (!team_any(nthr, again)) break;
    }
    norms();
  }
  __syncthreads();
  auto squared = [&](int i) {
    return i < rank && !(K::value(rows[i]) <= neg) ? static_cast<T>(K::value(rows[i])) * up * up : T(0);
  };
  if (tr != nullptr) {
    S *inv = rows;  // then their reciprocal roots
    for (int i = tid(); i < n; i += kThreads) {
      const T l = squared(i);
      const bool bad = !finite || !isfinite(l);
      if (bad) *tr->fail = STN_ENUMERIC;
      lam[i] = bad ? T(0) : l;
      if (i < rank) inv[i] = K::value(rows[i]) > 0 ? K::rsqrt(rows[i]) : K::of(0);
    }
    __syncthreads();
    for (int i = g; (i & ~3) < n; i += kGroups) {  // decreasing order, ties by index
      const T li = lam[min(i, n - 1)];
      int before = 0;
      for (int j = gl; j < n; j += kGroup) before += lam[j] > li || (lam[j] == li && j < i);
#pragma unroll
      for (int o = kGroup / 2; o > 0; o >>= 1) before += __shfl_xor_sync(0xffffffffu, before, o);
      if (gl == 0 && i < n) tr->perm[before] = i;
    }
    __syncthreads();
    if (*tr->fail) return 1;
    if (warp_id() == 0) {
      const int count = min(keep_count<T>(lam, tr->perm, n, tr->kmax, cutoff_, tr->delta), tr->kmax);
      if (lane_id() == 0) *tr->keep = count;
    }
    __syncthreads();
    const int keep = *tr->keep;
    if (warp_id() == kWarps - 1) {  // beside the others
      R share = 0;  // what was left: the columns without a pivot, whose norms the Jacobi has not touched
      if (left > 0)
        for (int c = lane_id(); c < n; c += 32) share += max(K::value(nr[c]), R(0));
      const double w = discarded_weight(lam, tr->perm, n, keep, static_cast<T>(share) * up * up);
      if (lane_id() == 0) *tr->discarded += w;
    } else {
      for (int e = tid(); e < n * keep; e += kThreads - 32) {
        const int c = e / n, i = e % n, row = tr->perm[c];
        cplx<T> v = cmake<T>(T(i == 0), 0);  // of a zero matrix
        if (row < rank) {
          const cplx<S> x = Bm[i * ld + row];
          v = cmake<T>(static_cast<T>(K::value(K::mul(x.re, inv[row]))), static_cast<T>(-K::value(K::mul(x.im, inv[row]))));
        }
        tr->vs[i * keep + c] = v;
        if (sizeof(T) == 4) tr->site[e] = cconj(v);
      }
    }
    __syncthreads();
    return keep;
  }
  for (int e = tid(); e < n * rank; e += kThreads) {
    const int i = e / n, c = e % n;
    const S s = rows[i];
    const cplx<S> x = Bm[c * ld + i];
    const S inv = K::value(s) > 0 ? K::rsqrt(s) : K::of(0);
    V[e] = cmake<T>(static_cast<T>(K::value(K::mul(x.re, inv))), static_cast<T>(-K::value(K::mul(x.im, inv))));
  }
  if (rank == 0)
    for (int c = tid(); c < n; c += kThreads) V[c] = cmake<T>(c == 0 ? T(1) : T(0), 0);
  for (int i = tid(); i < n; i += kThreads)
    lam[i] = finite ? squared(i) : static_cast<T>(__longlong_as_double(0x7ff8000000000000ll));
  __syncthreads();
  return rank;
}

STN_END
