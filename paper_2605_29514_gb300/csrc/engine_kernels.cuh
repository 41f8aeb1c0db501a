#pragma once
// Device code of the stabilizer-tensor-network simulation (sm_103a), shared by
// the translation units that instantiate it for complex64 (engine_f32.cu) and
// complex128 (engine_f64.cu), and by the allocation-free SVD
// (engine_noalloc.cu).
//
// One persistent CTA per shot slot walks the op list of a program segment
// (one syndrome round).  Clifford gates and Pauli noise update the inverse
// tableau held in shared memory (bit-exact integer row operations, Sec. IV A).
// A crosstalk rotation or a measurement pushes its Pauli through the tableau
// and acts on the shot's MPS as a bond-2 Pauli-string MPO; the touched span
// is then recompressed (Sec. IV B, Eq. 8) by a two-pass sweep:
//   left sweep   R_{k+1} = R factor of (R_k A'_k), R_a = identity since the
//                sites left of the span are left-canonical (Householder QR,
//                no Q formed); ||R_b A'_b||^2 is the squared norm of the new
//                state, which for a projector is the Born probability; a
//                matrix with no more rows than columns is its own R;
//   right sweep  C = R_k M_k = U Sigma V^dag (one-sided Jacobi); the kept
//                columns of V give the new right-canonical site and
//                M_{k-1} = A'_{k-1} (M_k V_keep) carries the rest to the left.
// Sigma holds the Schmidt values of the bond, so keeping the largest ones is
// the truncation of Eq. 8.  Small bonds are decomposed in shared memory (in
// pairs of floats on the complex64 path); large bonds take the Householder R
// factor of C and run Jacobi on its conjugate transpose, which converges in a
// few sweeps.  Dense work runs in complex T (float or
// double); norms, Born probabilities and log-probabilities in double.
#include <cuda_runtime.h>
#include <math.h>

#include <type_traits>

#include "../../include/stn.h"
#include "engine.h"

// The CTA size is a compile-time constant of the including file: 512 threads
// (one CTA per SM, all of its shared memory), or 256 for programs whose bonds
// stay small (kLightBond): barriers and reductions over half the warps are
// cheaper where a step's work fills neither, and two such CTAs fit an SM.  With
// one shot per SM, 256 threads took a d = 5 round at theta = 1e-3 from 120 to
// 107 ms, d = 7 from 194 to 174 ms, one d = 3 shot in complex128 from 23.7 to
// 20.7 ms; 128 threads were up to 10 % better at bonds of 4 and 10 % worse at 32.
#ifndef STN_CTA_THREADS
#define STN_CTA_THREADS 512
#endif
#if STN_CTA_THREADS == 512
#define STN_BEGIN namespace stn { inline namespace cta512 {
#else
#define STN_BEGIN namespace stn { inline namespace cta256 {
#endif
#define STN_END }}

STN_BEGIN

constexpr int kThreads = STN_CTA_THREADS;
constexpr bool kLight = kThreads < 512;

// ---------------------------------------------------------------------------
// complex arithmetic
template <typename T>
struct cplx {
  T re, im;
};
template <typename T>
__device__ __forceinline__ cplx<T> cmake(T r, T i) {
  cplx<T> c;
  c.re = r;
  c.im = i;
  return c;
}
template <typename T>
__device__ __forceinline__ cplx<T> cadd(cplx<T> a, cplx<T> b) {
  return cmake<T>(a.re + b.re, a.im + b.im);
}
template <typename T>
__device__ __forceinline__ cplx<T> cmul(cplx<T> a, cplx<T> b) {
  return cmake<T>(a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re);
}
template <typename T>
__device__ __forceinline__ cplx<T> cconj(cplx<T> a) {
  return cmake<T>(a.re, -a.im);
}
template <typename T>
__device__ __forceinline__ cplx<T> cscale(cplx<T> a, T s) {
  return cmake<T>(a.re * s, a.im * s);
}
// acc += a * b
template <typename T>
__device__ __forceinline__ void cfma(cplx<T> &acc, cplx<T> a, cplx<T> b) {
  acc.re = fma(a.re, b.re, acc.re);
  acc.re = fma(-a.im, b.im, acc.re);
  acc.im = fma(a.re, b.im, acc.im);
  acc.im = fma(a.im, b.re, acc.im);
}
template <typename T>
__device__ __forceinline__ T cabs2(cplx<T> a) {
  return a.re * a.re + a.im * a.im;
}
// |a|^2 in double from double components: in single precision the square of
// a component below about 1e-19 is a denormal or zero, which would make the
// norm of a tiny vector (and a reflector built from it) inaccurate.
template <typename T>
__device__ __forceinline__ double cabs2d(cplx<T> a) {
  const double re = static_cast<double>(a.re), im = static_cast<double>(a.im);
  return re * re + im * im;
}
// i^m
template <typename T>
__device__ __forceinline__ cplx<T> ipow(int m) {
  m &= 3;
  return m == 0 ? cmake<T>(1, 0) : m == 1 ? cmake<T>(0, 1) : m == 2 ? cmake<T>(-1, 0) : cmake<T>(0, -1);
}

template <typename T>
struct Eps;
template <>
struct Eps<float> {
  static constexpr float v = 5.96e-8f;
};
template <>
struct Eps<double> {
  static constexpr double v = 1.11e-16;
};

// Complex elements of shared memory for the one-sided Jacobi SVD (the matrix
// and its right singular vectors); larger problems run on global scratch.
template <typename T>
struct SvdSmem;
template <>
struct SvdSmem<float> {
  static constexpr int elems = 22528;
};
template <>
struct SvdSmem<double> {
  static constexpr int elems = 8192;
};
constexpr int kMaxVec = 1024;  // longest Householder vector (4 * largest bond)

constexpr int kTileElems = 2176;  // complex elements of a contraction's shared-memory tiles

// ---------------------------------------------------------------------------
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): two 32x32->64-bit
// multiplies per round, Weyl key schedule, ten rounds.
static __device__ __forceinline__ double philox_uniform(uint64_t seed, uint64_t shot, uint32_t ev) {
  uint32_t c0 = static_cast<uint32_t>(shot), c1 = static_cast<uint32_t>(shot >> 32);
  uint32_t c2 = ev, c3 = 0u;
  uint32_t k0 = static_cast<uint32_t>(seed), k1 = static_cast<uint32_t>(seed >> 32);
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    uint32_t lo0 = 0xD2511F53u * c0, hi0 = __umulhi(0xD2511F53u, c0);
    uint32_t lo1 = 0xCD9E8D57u * c2, hi1 = __umulhi(0xCD9E8D57u, c2);
    uint32_t n0 = hi1 ^ c1 ^ k0, n2 = hi0 ^ c3 ^ k1;
    c0 = n0;
    c1 = lo1;
    c2 = n2;
    c3 = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  uint64_t bits = (static_cast<uint64_t>(c0) << 21) ^ static_cast<uint64_t>(c1 >> 11);
  return static_cast<double>(bits) * 0x1.0p-53;
}


// ---------------------------------------------------------------------------
// CTA-wide helpers
static __device__ __forceinline__ int tid() { return threadIdx.x; }

// A pointer into dynamic shared memory that the compiler knows to be one: the
// larger routines are called, not inlined, and would use generic loads.
template <typename E>
__device__ __forceinline__ E *in_smem(const void *p) {
  extern __shared__ __align__(16) char smem_raw[];
  return reinterpret_cast<E *>(smem_raw + (static_cast<uint32_t>(__cvta_generic_to_shared(p)) -
                                           static_cast<uint32_t>(__cvta_generic_to_shared(smem_raw))));
}

// Sum of one double per thread over the CTA: a shuffle reduction per warp,
// then every thread adds the warps' partial sums (red: the first kThreads / 32
// of kRedDoubles doubles of shared memory).  Two barriers.
constexpr int kRedDoubles = 512;
static __device__ double block_sum(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) r += red[w];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------------------
// Complex64 GEMM on the fifth-generation tensor cores (tcgen05).  The CTA's
// tensor-memory accumulator (128 lanes x 128 FP32 columns: the real part of
// a 128 x 64 output tile, then its imaginary part), the two mbarriers the
// MMAs complete on and the shared-memory staging area of the operand tiles
// live in g_tc; a kernel that allocates the accumulator sets enabled.
//
// Each product is FP32-accurate from TF32 operands by the 3-term split
// (Ootomo and Yokota, 2022): x = x_hi + x_lo with both parts TF32, and
// A B ~ A_hi B_hi + A_hi B_lo + A_lo B_hi.  The complex product takes four
// real ones, Re C = Re A Re B + Im A (-Im B) and Im C = Re A Im B + Im A Re B,
// so every k step of 8 issues 6 MMAs per part (M = 128, N = 64, K = 8,
// kind::tf32) accumulated in FP32; the negated imaginary part is staged on
// the smaller B tile.  The k range goes in chunks of 16: the 128 x 16 A tile
// (4 arrays: Re and Im, head and tail) and the 64 x 16 B tile (6 arrays:
// Re, Im and -Im, head and tail) of a chunk are written to one of two
// staging buffers in the no-swizzle K-major core-matrix layout (core
// matrices of 8 rows x 16 bytes, 128 bytes apart along k, 512 bytes apart
// between 8-row groups), each thread storing whole 16-byte core-matrix rows
// so that a quarter warp fills one core matrix without bank conflicts.  After
// a proxy fence one thread issues the chunk's 24 MMAs and commits them to the
// buffer's mbarrier, and the CTA stages the next chunk into the other buffer
// while they run; a buffer is refilled only after a bounded wait on its
// barrier (on time-out the CTA's status becomes STN_ETIMEOUT and the product
// is abandoned).
struct TcState {
  uint64_t bar[2];  // mbarriers of the two staging buffers
  uint32_t tmem;    // tensor-memory address of the accumulator
  uint32_t phase;   // bit b: parity of bar[b]'s next completion
  int enabled;      // the kernel allocated tensor memory and staging space
  int failed;       // a bounded wait ran out
  float *stage;     // two staging buffers of kTcBufFloats floats
};
static __shared__ __align__(8) TcState g_tc;

constexpr int kTcM = 128, kTcN = 64, kTcK = 16;
constexpr int kTcAFloats = kTcM * kTcK, kTcBFloats = kTcN * kTcK;
constexpr int kTcBufFloats = 4 * kTcAFloats + 6 * kTcBFloats;
constexpr int kTcStageFloats = 2 * kTcBufFloats;
constexpr uint32_t kTcCols = 2 * kTcN;
constexpr long long kTcWaitLimit = 1ll << 24;
// kind::tf32, FP32 accumulator, both operands K-major, N = 64, M = 128
constexpr uint32_t kTcIdesc = (1u << 4) | (2u << 7) | (2u << 10) | (static_cast<uint32_t>(kTcN >> 3) << 17) |
                              (static_cast<uint32_t>(kTcM >> 4) << 24);

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// TF32 rounding (round to nearest, ties away) of an FP32 value, returned as
// the FP32 number it represents.
__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

// Float offset of the 16-byte core-matrix row (row, k = 4 kg .. 4 kg + 3)
// of a row x kTcK tile.
__device__ __forceinline__ int tc_row_offset(int row, int kg) {
  return (((row >> 3) * (kTcK / 4) + kg) * 128 + (row & 7) * 16) >> 2;
}

// Descriptor of the 8-wide k slice q of a staged tile (version 1, no
// swizzle): leading byte offset 128 (the next core matrix along k), stride
// byte offset kTcK / 4 x 128 (the next 8-row group).
__device__ __forceinline__ uint64_t tc_desc(const float *tile, int q) {
  const uint32_t a = smem_u32(tile) + static_cast<uint32_t>(q) * 256u;
  return static_cast<uint64_t>((a >> 4) & 0x3FFF) | (static_cast<uint64_t>(128 >> 4) << 16) |
         (static_cast<uint64_t>((kTcK / 4 * 128) >> 4) << 32) | (static_cast<uint64_t>(1) << 46);
}

__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n"
      :
      : "r"(d), "l"(a), "l"(b), "r"(kTcIdesc), "r"(acc));
}

__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t phase) {
  for (long long it = 0; it < kTcWaitLimit; ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(phase)
        : "memory");
    if (done) return true;
  }
  return false;
}

// Tensor memory and barriers of a CTA that runs tensor-core GEMMs (CTA-wide;
// warp 0 allocates).  stage: kTcStageFloats floats of shared memory, 16-byte
// aligned, free whenever a GEMM runs.
static __device__ void tc_setup(float *stage) {
  if ((threadIdx.x >> 5) == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&g_tc.tmem)),
                 "r"(kTcCols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&g_tc.bar[0])));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_u32(&g_tc.bar[1])));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    g_tc.phase = 0;
    g_tc.failed = 0;
    g_tc.stage = stage;
    g_tc.enabled = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
}

static __device__ void tc_teardown() {
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  if ((threadIdx.x >> 5) == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(g_tc.tmem), "r"(kTcCols));
}

// Static shared memory starts with whatever the SM's previous kernel left
// there, so a kernel without tensor memory clears both flags.
static __device__ __forceinline__ void tc_disable() {
  if (threadIdx.x == 0) {
    g_tc.enabled = 0;
    g_tc.failed = 0;
  }
  __syncthreads();
}

static_assert(kLight || kThreads == 512, "the tensor-core staging and epilogue map 512 threads onto the tiles");

__device__ __forceinline__ void st_f4(float *p, float a, float b, float c, float d) {
  *reinterpret_cast<float4 *>(p) = make_float4(a, b, c, d);
}

// Stages the k chunk k0 .. k0 + kTcK - 1 of rows i0 .. i0 + 127 of op(A) and
// columns j0 .. j0 + 63 of op(B) into the staging buffer buf (zero outside
// the matrices).  Item f of a tile is the core-matrix row (row, kg) with
// row = (f & 7) + 8 (f >> 5) and kg = (f >> 3) & 3, so that the eight
// threads of a quarter warp write the eight rows of one core matrix.
template <int TA, int TB>
static __device__ __forceinline__ void tc_stage(float *buf, int M, int N, int K, const cplx<float> *A, int lda,
                                                const cplx<float> *B, int ldb, int i0, int j0, int k0) {
  for (int e = threadIdx.x; e < 4 * (kTcM + kTcN); e += kThreads) {
    const bool isA = e < 4 * kTcM;  // warp-uniform: 4 kTcM is a multiple of kThreads
    const int f = isA ? e : e - 4 * kTcM;
    const int row = (f & 7) | ((f >> 5) << 3), kg = (f >> 3) & 3;
    float rh[4], rl[4], ih[4], il[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int gk = k0 + 4 * kg + u;
      cplx<float> v = cmake<float>(0.f, 0.f);
      if (isA) {
        const int gi = i0 + row;
        if (gi < M && gk < K)
          v = TA == 0 ? A[static_cast<int64_t>(gi) * lda + gk] : cconj(A[static_cast<int64_t>(gk) * lda + gi]);
      } else {
        const int gj = j0 + row;
        if (gj < N && gk < K)
          v = TB == 0 ? B[static_cast<int64_t>(gk) * ldb + gj] : cconj(B[static_cast<int64_t>(gj) * ldb + gk]);
      }
      rh[u] = tf32_round(v.re);
      rl[u] = tf32_round(v.re - rh[u]);
      ih[u] = tf32_round(v.im);
      il[u] = tf32_round(v.im - ih[u]);
    }
    const int o = tc_row_offset(row, kg);
    float *dst = isA ? buf + o : buf + 4 * kTcAFloats + o;
    const int s = isA ? kTcAFloats : kTcBFloats;
    st_f4(dst, rh[0], rh[1], rh[2], rh[3]);
    st_f4(dst + s, rl[0], rl[1], rl[2], rl[3]);
    st_f4(dst + 2 * s, ih[0], ih[1], ih[2], ih[3]);
    st_f4(dst + 3 * s, il[0], il[1], il[2], il[3]);
    if (!isA) {
      st_f4(dst + 4 * s, -ih[0], -ih[1], -ih[2], -ih[3]);
      st_f4(dst + 5 * s, -il[0], -il[1], -il[2], -il[3]);
    }
  }
}

// The 24 MMAs of one staged chunk (two k slices of 8) into the real and
// imaginary accumulators; the first slice of a tile overwrites them.
static __device__ __forceinline__ void tc_issue_chunk(const float *buf, uint32_t tm_re, uint32_t tm_im, bool first) {
  const float *Ab = buf, *Bb = buf + 4 * kTcAFloats;
#pragma unroll
  for (int q = 0; q < kTcK / 8; ++q) {
    const uint32_t acc = (!first || q > 0) ? 1u : 0u;
    const uint64_t a_rh = tc_desc(Ab, q), a_rl = tc_desc(Ab + kTcAFloats, q), a_ih = tc_desc(Ab + 2 * kTcAFloats, q),
                   a_il = tc_desc(Ab + 3 * kTcAFloats, q);
    const uint64_t b_rh = tc_desc(Bb, q), b_rl = tc_desc(Bb + kTcBFloats, q), b_ih = tc_desc(Bb + 2 * kTcBFloats, q),
                   b_il = tc_desc(Bb + 3 * kTcBFloats, q), b_nh = tc_desc(Bb + 4 * kTcBFloats, q),
                   b_nl = tc_desc(Bb + 5 * kTcBFloats, q);
    tc_mma(tm_re, a_rh, b_rh, acc);  // Re A Re B
    tc_mma(tm_re, a_rh, b_rl, 1u);
    tc_mma(tm_re, a_rl, b_rh, 1u);
    tc_mma(tm_re, a_ih, b_nh, 1u);   // Im A (-Im B)
    tc_mma(tm_re, a_ih, b_nl, 1u);
    tc_mma(tm_re, a_il, b_nh, 1u);
    tc_mma(tm_im, a_rh, b_ih, acc);  // Re A Im B
    tc_mma(tm_im, a_rh, b_il, 1u);
    tc_mma(tm_im, a_rl, b_ih, 1u);
    tc_mma(tm_im, a_ih, b_rh, 1u);   // Im A Re B
    tc_mma(tm_im, a_ih, b_rl, 1u);
    tc_mma(tm_im, a_il, b_rh, 1u);
  }
}

// Kept out of line so that its registers do not weigh on the callers'.
template <int TA, int TB>
static __device__ __noinline__ void cgemm_tc(int M, int N, int K, cplx<float> alpha, const cplx<float> *A, int lda,
                                             const cplx<float> *B, int ldb, cplx<float> beta, cplx<float> *C,
                                             int ldc) {
  float *st = g_tc.stage;
  const uint32_t tm_re = g_tc.tmem, tm_im = g_tc.tmem + kTcN;
  const uint32_t bar0 = smem_u32(&g_tc.bar[0]), bar1 = smem_u32(&g_tc.bar[1]);
  uint32_t phase = g_tc.phase;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool beta0 = beta.re == 0.f && beta.im == 0.f;
  const int nk = (K + kTcK - 1) / kTcK;
  bool ok = true;
  uint32_t pending = 0;  // bit b: buffer b holds committed MMAs not yet waited on
  for (int i0 = 0; i0 < M && ok; i0 += kTcM) {
    for (int j0 = 0; j0 < N && ok; j0 += kTcN) {
      for (int kc = 0; kc < nk; ++kc) {
        const int b = kc & 1;
        bool waited = true;
        if (pending & (1u << b)) {  // the MMAs of chunk kc - 2 still read this buffer
          waited = tc_wait(b ? bar1 : bar0, (phase >> b) & 1u);
          phase ^= 1u << b;
          pending &= ~(1u << b);
        }
        float *buf = st + b * kTcBufFloats;
        if (waited) tc_stage<TA, TB>(buf, M, N, K, A, lda, B, ldb, i0, j0, kc * kTcK);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n");
        const int failed = __syncthreads_or(waited ? 0 : 1);
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        if (failed) {
          ok = false;
          break;
        }
        if (threadIdx.x == 0) {
          tc_issue_chunk(buf, tm_re, tm_im, kc == 0);
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                           b ? bar1 : bar0)
                       : "memory");
        }
        pending |= 1u << b;
      }
      if (!ok) break;
      // the tile's last MMAs (and the older chunk in the other buffer)
      bool waited = true;
#pragma unroll
      for (int b = 0; b < 2; ++b)
        if (pending & (1u << b)) {
          waited = tc_wait(b ? bar1 : bar0, (phase >> b) & 1u) && waited;
          phase ^= 1u << b;
        }
      pending = 0;
      asm volatile("tcgen05.fence::after_thread_sync;\n");
      if (__syncthreads_or(waited ? 0 : 1)) {
        ok = false;
        break;
      }
      // epilogue: warp w reads lanes 32 (w % 4) .. + 31, columns 16 (w / 4) .. + 15,
      // eight at a time
      const int quarter = warp & 3;
      const uint32_t lane_off = static_cast<uint32_t>(32 * quarter) << 16;
      const int row = i0 + 32 * quarter + lane;
#pragma unroll
      for (int half = 0; half < 2; ++half) {
        const int cb = 16 * (warp >> 2) + 8 * half;
        uint32_t vr[8], vi[8];
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                     : "=r"(vr[0]), "=r"(vr[1]), "=r"(vr[2]), "=r"(vr[3]), "=r"(vr[4]), "=r"(vr[5]), "=r"(vr[6]),
                       "=r"(vr[7])
                     : "r"(tm_re + lane_off + cb));
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                     : "=r"(vi[0]), "=r"(vi[1]), "=r"(vi[2]), "=r"(vi[3]), "=r"(vi[4]), "=r"(vi[5]), "=r"(vi[6]),
                       "=r"(vi[7])
                     : "r"(tm_im + lane_off + cb));
        asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
        if (row < M) {
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const int col = j0 + cb + c;
            if (col >= N) continue;
            cplx<float> v = cmul(alpha, cmake<float>(__uint_as_float(vr[c]), __uint_as_float(vi[c])));
            cplx<float> *dst = &C[static_cast<int64_t>(row) * ldc + col];
            if (!beta0) v = cadd(v, cmul(beta, *dst));
            *dst = v;
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncthreads();
      asm volatile("tcgen05.fence::after_thread_sync;\n");
    }
  }
  if (!ok) {  // give the MMAs in flight a last bounded chance to land, then report
#pragma unroll
    for (int b = 0; b < 2; ++b)
      if (pending & (1u << b)) {
        tc_wait(b ? bar1 : bar0, (phase >> b) & 1u);
        phase ^= 1u << b;
      }
    if (threadIdx.x == 0) g_tc.failed = 1;
  }
  if (threadIdx.x == 0) g_tc.phase = phase;
  __syncthreads();
}

// Contractions of small bonds, straight from global memory (the L1 holds the
// operands): thread t owns column t % N of U output rows t / N + u (kThreads
// / N), so a row of B is read once for U products and nothing is padded.  The
// shared-memory tiles below round every product up to 64 x 64 x 16.  For an
// 8 x 8 x 8 complex128 product that is 128 times its arithmetic, on a pipe of
// two FP64 FMAs a clock: 68 us in tiles, 8 us here, which is the launch's time;
// by one CTA 200^3 takes 13.4 ms in tiles and 8.3 ms here, so complex128 always comes
// here (N <= 512 in a sweep; a wider product runs in tiles).  In complex64 the
// tiles' arithmetic is cheap but their barriers are not: up to 2^16 products
// the direct form is faster (one d = 5 round at cap 32: 439 ms in tiles, 406
// ms), beyond that the operands' reuse in shared memory wins (64^3: 15 us in
// tiles, 22 us).
template <typename T>
static __device__ __forceinline__ bool gemm_direct(int M, int N, int K) {
  if (N > kThreads) return false;
  return sizeof(T) == 8 || static_cast<int64_t>(M) * N * K <= 65536;
}

template <typename T, int TA, int TB, int U>
static __device__ __forceinline__ void cgemm_rows(int M, int N, int K, cplx<T> alpha, const cplx<T> *A, int lda,
                                                  const cplx<T> *B, int ldb, cplx<T> beta, cplx<T> *C, int ldc) {
  const int rp = kThreads / N, j = threadIdx.x % N, ty = threadIdx.x / N;
  if (ty < rp) {
    for (int i0 = ty; i0 < M; i0 += rp * U) {
      cplx<T> acc[U];
#pragma unroll
      for (int u = 0; u < U; ++u) acc[u] = cmake<T>(0, 0);
#pragma unroll 4
      for (int k = 0; k < K; ++k) {
        const cplx<T> b = TB == 0 ? B[static_cast<int64_t>(k) * ldb + j] : cconj(B[static_cast<int64_t>(j) * ldb + k]);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int i = min(i0 + u * rp, M - 1);  // a row past the end repeats the last one, unused
          const cplx<T> a = TA == 0 ? A[static_cast<int64_t>(i) * lda + k] : cconj(A[static_cast<int64_t>(k) * lda + i]);
          cfma(acc[u], a, b);
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * rp;
        if (i >= M) break;
        cplx<T> *c = &C[static_cast<int64_t>(i) * ldc + j];
        cplx<T> v = cmul(alpha, acc[u]);
        if (beta.re != T(0) || beta.im != T(0)) v = cadd(v, cmul(beta, *c));
        *c = v;
      }
    }
  }
  __syncthreads();
}

// Larger products in shared-memory tiles of kTY MR x 64 outputs, a slice of
// kTileK of the k range at a time: thread (ty, tx) of a kTY x 16 grid owns rows
// ty + kTY a and columns tx + 16 b, so a k step reads MR + 4 elements, which the
// lanes of a warp read without conflicts, for 4 MR products.  The next slice is fetched from global memory into
// registers while the present one is multiplied.
constexpr int kTileK = 8;

template <typename T, int TA, int TB, int MR>
static __device__ __forceinline__ void cgemm_tiles(int M, int N, int K, cplx<T> alpha, const cplx<T> *A, int lda,
                                                   const cplx<T> *B, int ldb, cplx<T> beta, cplx<T> *C, int ldc,
                                                   cplx<T> *tile) {
  constexpr int kTY = kThreads / 16, RM = kTY * MR, RN = 64, LA = RM + 2, LB = RN + 2;  // padded rows of a slice
  constexpr int NA = RM * kTileK / kThreads, NB = RN * kTileK / kThreads;
  static_assert(NA * kThreads == RM * kTileK && NB * kThreads == RN * kTileK && kTileK * (LA + LB) <= kTileElems, "tile");
  cplx<T> *As = in_smem<cplx<T>>(tile), *Bs = As + kTileK * LA;
  const int ty = threadIdx.x / 16, tx = threadIdx.x % 16;
  for (int i0 = 0; i0 < M; i0 += RM)
    for (int j0 = 0; j0 < N; j0 += RN) {
      cplx<T> acc[MR][4], pa[NA], pb[NB];
#pragma unroll
      for (int a = 0; a < MR; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) acc[a][b] = cmake<T>(0, 0);
      auto fetch = [&](int k0) {
#pragma unroll
        for (int r = 0; r < NA; ++r) {
          const int e = threadIdx.x + r * kThreads;
          const int k = TA == 0 ? e % kTileK : e / RM, i = TA == 0 ? e / kTileK : e % RM;
          const int gi = i0 + i, gk = k0 + k;
          pa[r] = cmake<T>(0, 0);
          if (gi < M && gk < K)
            pa[r] = TA == 0 ? A[static_cast<int64_t>(gi) * lda + gk] : cconj(A[static_cast<int64_t>(gk) * lda + gi]);
        }
#pragma unroll
        for (int r = 0; r < NB; ++r) {
          const int e = threadIdx.x + r * kThreads;
          const int k = TB == 0 ? e / RN : e % kTileK, j = TB == 0 ? e % RN : e / kTileK;
          const int gj = j0 + j, gk = k0 + k;
          pb[r] = cmake<T>(0, 0);
          if (gj < N && gk < K)
            pb[r] = TB == 0 ? B[static_cast<int64_t>(gk) * ldb + gj] : cconj(B[static_cast<int64_t>(gj) * ldb + gk]);
        }
      };
      fetch(0);
      for (int k0 = 0; k0 < K; k0 += kTileK) {
#pragma unroll
        for (int r = 0; r < NA; ++r) {
          const int e = threadIdx.x + r * kThreads;
          if (TA == 0) As[(e % kTileK) * LA + e / kTileK] = pa[r];
          else As[(e / RM) * LA + e % RM] = pa[r];
        }
#pragma unroll
        for (int r = 0; r < NB; ++r) {
          const int e = threadIdx.x + r * kThreads;
          if (TB == 0) Bs[(e / RN) * LB + e % RN] = pb[r];
          else Bs[(e % kTileK) * LB + e / kTileK] = pb[r];
        }
        __syncthreads();
        if (k0 + kTileK < K) fetch(k0 + kTileK);
#pragma unroll
        for (int k = 0; k < kTileK; ++k) {
          cplx<T> av[MR], bv[4];
#pragma unroll
          for (int a = 0; a < MR; ++a) av[a] = As[k * LA + ty + kTY * a];
#pragma unroll
          for (int b = 0; b < 4; ++b) bv[b] = Bs[k * LB + tx + 16 * b];
#pragma unroll
          for (int a = 0; a < MR; ++a)
#pragma unroll
            for (int b = 0; b < 4; ++b) cfma(acc[a][b], av[a], bv[b]);
        }
        __syncthreads();
      }
#pragma unroll
      for (int a = 0; a < MR; ++a) {
        const int gi = i0 + ty + kTY * a;
        if (gi >= M) continue;
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const int gj = j0 + tx + 16 * b;
          if (gj >= N) continue;
          cplx<T> *c = &C[static_cast<int64_t>(gi) * ldc + gj];
          cplx<T> v = cmul(alpha, acc[a][b]);
          if (beta.re != T(0) || beta.im != T(0)) v = cadd(v, cmul(beta, *c));
          *c = v;
        }
      }
    }
  __syncthreads();
}

// C = alpha * op(A) op(B) + beta * C, all row-major, op = identity (0) or
// conjugate transpose (1).  op(A) is M x K, op(B) is K x N.  Complex64
// products large enough to fill the tensor-core tiles run cgemm_tc when the
// kernel enabled it; the rest (and complex128) run on the CUDA cores below.
template <typename T, int TA, int TB>
static __device__ __noinline__ void cgemm(int M, int N, int K, cplx<T> alpha, const cplx<T> *A, int lda,
                      const cplx<T> *B, int ldb, cplx<T> beta, cplx<T> *C, int ldc,
                      cplx<T> *tile) {
  if constexpr (sizeof(T) == 4 && !kLight) {
    if (g_tc.enabled && M >= 64 && N >= 32 && K >= kTcK) {
      cgemm_tc<TA, TB>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
      return;
    }
  }
  if (gemm_direct<T>(M, N, K)) {
    const int rp = kThreads / N;
    if (M <= rp) cgemm_rows<T, TA, TB, 1>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    else if (M <= 2 * rp) cgemm_rows<T, TA, TB, 2>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    else cgemm_rows<T, TA, TB, 4>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc);
    return;
  }
  if (M <= 64) cgemm_tiles<T, TA, TB, 2>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, tile);
  else cgemm_tiles<T, TA, TB, 4>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, tile);
}

static __device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }
static __device__ __forceinline__ int lane_id() { return threadIdx.x & 31; }
constexpr int kWarps = kThreads / 32;

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

constexpr int kMaxSweepsF = 15, kMaxSweepsD = 20;  // Jacobi

STN_END

#include "small_bond.cuh"

STN_BEGIN

// A dense problem that is called alone may be shared by the CTAs of a cluster
// (CL): its matrix lies in global memory, and phases that write it end in
// share_sync, whose release and acquire order that memory over the cluster.
template <bool CL>
__device__ __forceinline__ int share_rank() {
  int r = 0;
  if constexpr (CL) asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
template <bool CL>
__device__ __forceinline__ int share_size() {
  int r = 1;
  if constexpr (CL) asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
template <bool CL>
__device__ __forceinline__ void share_sync() {
  if constexpr (CL) {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;\n" ::: "memory");
  } else {
    __syncthreads();
  }
}
// An int of the shared memory of CTA `rank` of the cluster, at this CTA's address p.
template <bool CL>
__device__ __forceinline__ int share_load(const int *p, int rank) {
  if constexpr (!CL) return *p;
  uint32_t a;
  int v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
template <bool CL>
__device__ __forceinline__ void share_store(int *p, int rank, int v) {
  if constexpr (!CL) {
    *p = v;
  } else {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
    asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
  }
}

// Householder QR of B (m x n, row-major, leading dimension ld), in place: on
// return rows 0..min(m,n)-1 hold R (upper trapezoidal) and the rest is zero.
// Each step uses the Hermitian reflector P = I - 2 u u^dag with
// P x = gamma e_1, gamma = -(x_0/|x_0|) ||x||.  Blocked by panels of nb
// columns: a panel is copied to shared memory (pbuf) and factored there,
// its reflectors u_1..u_nb are kept as the columns of V, and the product
// P_nb ... P_1 = I - V T^dag V^dag (compact WY form, T upper triangular with
// T_kk = 2, T[0:k, k] = -2 T[0:k, 0:k] V[:, 0:k]^dag u_k) is applied to the
// trailing columns at once (qr_trailing), so the trailing matrix is
// read and written twice per panel rather than per column.  pbuf needs
// m (nb + 1) + 2 nb^2 complex elements (nb is reduced to fit).  CTA-wide, or over
// a cluster: every CTA factors the panel for itself, the first one writes it back,
// and the trailing columns are split.  R is the same to the last bit either way:
// row j of R carries the phase of x_j, known to eps ||x|| / |x_j| only, so sums in
// another order would move single elements of a large R by 1e-3.
constexpr int kQrPanel = 16;

static __device__ __forceinline__ int qr_panel_width(int m, int pbuf_elems) {
  int nb = kQrPanel;
  while (nb > 1 && static_cast<int64_t>(m) * (nb + 1) + 2 * nb * nb > pbuf_elems) --nb;
  return nb;
}

// T of the compact WY form of a panel's reflectors (columns of Vp, row-major
// [mr][ldv], u_b zero above row b): T upper triangular, T_kk = 2,
// T[0:k, k] = -2 T[0:k, 0:k] (V[:, 0:k]^dag u_k).  G is scratch.  CTA-wide.
template <typename T>
static __device__ void wy_t_factor(int mr, int jb, int nb, int ldv, const cplx<T> *Vp, cplx<T> *Tm, cplx<T> *G) {
  for (int pr = warp_id(); pr < jb * jb; pr += kWarps) {
    const int a = pr / jb, b = pr % jb;
    if (a >= b) continue;
    T gr = 0, gi = 0;
    for (int i = b + lane_id(); i < mr; i += 32) {  // u_b vanishes above row b
      const cplx<T> x = Vp[i * ldv + a], y = Vp[i * ldv + b];
      gr += x.re * y.re + x.im * y.im;
      gi += x.re * y.im - x.im * y.re;
    }
    gr = warp_sum(gr);
    gi = warp_sum(gi);
    if (lane_id() == 0) G[a * nb + b] = cmake<T>(gr, gi);
  }
  __syncthreads();
  if (warp_id() == 0) {  // a lane owns a row of T
    const int a = lane_id();
    for (int k = 0; k < jb; ++k) {
      cplx<T> acc = cmake<T>(0, 0);
      if (a < k)
        for (int b = a; b < k; ++b) cfma(acc, Tm[a * nb + b], G[b * nb + k]);
      if (a < k) Tm[a * nb + k] = cscale(acc, T(-2));
      if (a == k) Tm[k * nb + k] = cmake<T>(2, 0);
    }
  }
  __syncthreads();
}

// Trailing columns of a panel: b <- b - V (T^dag (V^dag b)).  The columns go to
// the warps in groups of cpw consecutive ones (coalesced row reads).  The ns G
// lanes that share a column split w = V^dag b: slice s sums over the rows s, s +
// ns, ..., for the reflectors of one of G groups; the slices' partials are summed
// by shuffles and the groups' values exchanged, and then the lanes split the rows
// of the update.  w and the update depend on ns but not on G, which spreads a
// column over more lanes without another order of summation.  Rows go several at
// a time so that their loads are in flight together.  A cluster's CTAs have lanes
// to spare: with G = 4 or 8 the R factor of 512 x 250 in complex64 takes 1.36 ms;
// more slices instead (ns = 8) took 1.57 ms and gave an R with other phases.
template <typename T, int G>
static __device__ __forceinline__ void qr_trailing(int mr, int n, int j0, int jb, int nb, int ldv, const cplx<T> *Vp,
                                                   const cplx<T> *Tm, cplx<T> *B, int ld, int ns, int warp,
                                                   int warps) {
  constexpr int KW = kQrPanel / G;  // reflectors of a lane
  constexpr int U = G == 1 ? 4 : 64 / static_cast<int>(sizeof(T));  // rows in flight in w
  const int cpw = 32 / (ns * G), part = lane_id() / cpw, s = part % ns, k0 = part / ns * KW;
  for (int cb = j0 + jb + warp * cpw; cb < n; cb += warps * cpw) {  // warp-uniform trip count
    const int c = cb + lane_id() % cpw;
    const bool valid = c < n;
    cplx<T> own[KW], all[G == 1 ? 1 : kQrPanel], *const w = G == 1 ? own : all;
#pragma unroll
    for (int k = 0; k < KW; ++k) own[k] = cmake<T>(0, 0);
    if (valid) {
      int i = s;
      for (; i + (U - 1) * ns < mr; i += U * ns) {
        cplx<T> b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) b[u] = B[static_cast<int64_t>(j0 + i + u * ns) * ld + c];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
          for (int k = 0; k < KW; ++k)
            if (k0 + k < jb) cfma(own[k], cconj(Vp[(i + u * ns) * ldv + k0 + k]), b[u]);
      }
      for (; i < mr; i += ns) {
        const cplx<T> b = B[static_cast<int64_t>(j0 + i) * ld + c];
#pragma unroll
        for (int k = 0; k < KW; ++k)
          if (k0 + k < jb) cfma(own[k], cconj(Vp[i * ldv + k0 + k]), b);
      }
    }
    for (int off = cpw; off < cpw * ns; off *= 2)
#pragma unroll
      for (int k = 0; k < KW; ++k)
        if (G > 1 || k < jb) {
          own[k].re += __shfl_xor_sync(0xffffffffu, own[k].re, off);
          own[k].im += __shfl_xor_sync(0xffffffffu, own[k].im, off);
        }
    // every lane gets the groups' values, in order
    auto exchange = [&]() {
      if constexpr (G > 1) {
        const int first = lane_id() % (cpw * ns);
#pragma unroll
        for (int k = 0; k < kQrPanel; ++k) {
          const int from = first + k / KW * (cpw * ns);
          w[k] = cmake<T>(__shfl_sync(0xffffffffu, own[k % KW].re, from), __shfl_sync(0xffffffffu, own[k % KW].im, from));
        }
      }
    };
    exchange();
    // w <- T^dag w, highest index first: w'[a] = sum_{b<=a} conj(T[b][a]) w[b]
#pragma unroll
    for (int k = KW - 1; k >= 0; --k) {
      const int a = k0 + k;
      if (a >= jb) continue;
      cplx<T> acc = cmake<T>(0, 0);
#pragma unroll
      for (int b = 0; b < kQrPanel; ++b)
        if (b <= a) cfma(acc, cconj(Tm[b * nb + a]), w[b]);
      own[k] = acc;
    }
    exchange();
    if (valid) {
      const int step = ns * G;
      int i = part;
      for (; i + 3 * step < mr; i += 4 * step) {
        cplx<T> b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = B[static_cast<int64_t>(j0 + i + u * step) * ld + c];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
#pragma unroll
          for (int k = 0; k < kQrPanel; ++k)
            if (k < jb) {
              const cplx<T> t = cmul(Vp[(i + u * step) * ldv + k], w[k]);
              b[u] = cmake<T>(b[u].re - t.re, b[u].im - t.im);
            }
          B[static_cast<int64_t>(j0 + i + u * step) * ld + c] = b[u];
        }
      }
      for (; i < mr; i += step) {
        cplx<T> &bref = B[static_cast<int64_t>(j0 + i) * ld + c];
        cplx<T> acc = bref;
#pragma unroll
        for (int k = 0; k < kQrPanel; ++k)
          if (k < jb) {
            const cplx<T> t = cmul(Vp[i * ldv + k], w[k]);
            acc = cmake<T>(acc.re - t.re, acc.im - t.im);
          }
        bref = acc;
      }
    }
  }
}

// With vstore (row-major m x min(m,n)), the reflectors are also kept there
// (column j holds u_j in rows j..m-1; rows above are not written) so that
// form_q can build Q explicitly.
template <typename T, bool CL = false>
static __device__ __noinline__ void qr_r_inplace(int m, int n, cplx<T> *B, int ld, cplx<T> *pbuf_, int pbuf_elems,
                                                 cplx<T> *vstore = nullptr) {
  cplx<T> *pbuf = in_smem<cplx<T>>(pbuf_);
  const int steps = min(m, n);
  const int nb = qr_panel_width(m, pbuf_elems);
  // rows of the panel padded to an odd number of elements, so that a column
  // walked by consecutive threads spreads over the shared-memory banks
  const int ldv = nb + 1;
  cplx<T> *Vp = pbuf;                                    // [(m - j0)][ldv], row-major
  cplx<T> *Tm = pbuf + static_cast<int64_t>(m) * ldv;  // [nb][nb]
  cplx<T> *G = Tm + nb * nb;                            // [nb][nb], G[a][b] = u_a^dag u_b
  for (int j0 = 0; j0 < steps; j0 += nb) {
    const int jb = min(nb, steps - j0);
    const int mr = m - j0;
    for (int e = tid(); e < mr * jb; e += kThreads) {
      const int i = e / jb, c = e % jb;
      Vp[i * ldv + c] = B[static_cast<int64_t>(j0 + i) * ld + j0 + c];
    }
    share_sync<CL>();
    // Panel: a warp owns a column (two of a 256-thread CTA's).  The warp that has
    // brought column jj + 1 up to date forms its reflector at once, in place, while
    // the others still update theirs, so a column takes one barrier.  (Norm by the
    // whole CTA, scalars by one thread in double, four barriers: about 12,000
    // cycles a column.)
    const bool writes = share_rank<CL>() == 0;
    auto reflect = [&](int jj) {
      const Reflector<T> h = column_reflector(Vp + jj, ldv, jj, mr, true);
      cplx<T> *out = B + static_cast<int64_t>(j0) * ld + j0 + jj;
      for (int i = lane_id(); i < mr; i += 32) {
        cplx<T> &x = Vp[i * ldv + jj];
        if (i < jj) {  // rows above the diagonal are final R entries
          if (writes) out[static_cast<int64_t>(i) * ld] = x;
          x = cmake<T>(0, 0);
        } else {
          x = h.vector(x, i == jj);
          if (writes) out[static_cast<int64_t>(i) * ld] = i == jj ? h.diagonal() : cmake<T>(0, 0);
        }
      }
      __syncwarp();
    };
    if (warp_id() == 0) reflect(0);
    __syncthreads();
    for (int jj = 0; jj + 1 < jb; ++jj) {
      for (int c = warp_id(); c < jb; c += kWarps) {
        if (c <= jj) continue;  // b <- b - 2 u (u^dag b)
        T sr = 0, si = 0;
#pragma unroll 4
        for (int i = jj + lane_id(); i < mr; i += 32) {
          const cplx<T> u = Vp[i * ldv + jj], b = Vp[i * ldv + c];
          sr += u.re * b.re + u.im * b.im;
          si += u.re * b.im - u.im * b.re;
        }
        sr = warp_sum(sr);
        si = warp_sum(si);
        const cplx<T> s2 = cmake<T>(T(2) * sr, T(2) * si);
#pragma unroll 4
        for (int i = jj + lane_id(); i < mr; i += 32) {
          const cplx<T> t = cmul(Vp[i * ldv + jj], s2);
          cplx<T> &b = Vp[i * ldv + c];
          b = cmake<T>(b.re - t.re, b.im - t.im);
        }
        __syncwarp();
        if (c == jj + 1) reflect(c);
      }
      __syncthreads();
    }
    if (vstore != nullptr && writes)
      for (int e = tid(); e < mr * jb; e += kThreads) {
        const int i = e / jb, c = e % jb;
        vstore[static_cast<int64_t>(j0 + i) * steps + j0 + c] = Vp[i * ldv + c];
      }
    if (j0 + jb >= n) {  // no trailing columns
      share_sync<CL>();
      continue;
    }
    wy_t_factor<T>(mr, jb, nb, ldv, Vp, Tm, G);
    {
      // the slices of one CTA whatever the number of CTAs, so that R does not depend on it
      const int nt = n - j0 - jb, ranks = share_size<CL>();
      int ns = 1;
      while (ns < 8 && nt * 2 * ns <= kThreads) ns *= 2;
      const int warp = warp_id() * ranks + share_rank<CL>(), warps = kWarps * ranks;
      if constexpr (CL) {  // as many lanes as a warp has for its columns
        if (ns == 8) qr_trailing<T, 4>(mr, n, j0, jb, nb, ldv, Vp, Tm, B, ld, ns, warp, warps);
        else qr_trailing<T, 8>(mr, n, j0, jb, nb, ldv, Vp, Tm, B, ld, ns, warp, warps);
      } else {
        qr_trailing<T, 1>(mr, n, j0, jb, nb, ldv, Vp, Tm, B, ld, ns, warp, warps);
      }
    }
    share_sync<CL>();
  }
}

// Explicit Q (m x steps, row-major) of a Householder QR whose reflectors
// qr_r_inplace kept in vstore: Q = P_1 ... P_steps [I; 0], built panel by
// panel from the last, each panel applied as I - V T V^dag to the columns at
// or right of it (the columns left of panel p are unit vectors its
// reflectors do not touch).  Same shared-memory needs as qr_r_inplace.
template <typename T>
static __device__ __noinline__ void form_q(int m, int steps, const cplx<T> *vstore, cplx<T> *Q, cplx<T> *pbuf_,
                                           int pbuf_elems) {
  cplx<T> *pbuf = in_smem<cplx<T>>(pbuf_);
  const int nb = qr_panel_width(m, pbuf_elems);
  const int ldv = nb + 1;
  cplx<T> *Vp = pbuf;
  cplx<T> *Tm = pbuf + static_cast<int64_t>(m) * ldv;
  cplx<T> *G = Tm + nb * nb;
  for (int64_t e = tid(); e < static_cast<int64_t>(m) * steps; e += kThreads) {
    const int i = static_cast<int>(e / steps), c = static_cast<int>(e % steps);
    Q[e] = cmake<T>(i == c ? T(1) : T(0), 0);
  }
  const int npan = (steps + nb - 1) / nb;
  for (int p = npan - 1; p >= 0; --p) {
    const int j0 = p * nb, jb = min(nb, steps - j0), mr = m - j0;
    for (int e = tid(); e < mr * nb; e += kThreads) {
      const int i = e / nb, c = e % nb;
      // u_c is zero above its own row; rows above were never written
      Vp[i * ldv + c] = (c < jb && i >= c) ? vstore[static_cast<int64_t>(j0 + i) * steps + j0 + c] : cmake<T>(0, 0);
    }
    __syncthreads();
    wy_t_factor<T>(mr, jb, nb, ldv, Vp, Tm, G);
    for (int c = j0 + tid(); c < steps; c += kThreads) {
      cplx<T> w[kQrPanel];
#pragma unroll
      for (int k = 0; k < kQrPanel; ++k) w[k] = cmake<T>(0, 0);
      int i = 0;
      for (; i + 4 <= mr; i += 4) {
        cplx<T> q[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) q[u] = Q[static_cast<int64_t>(j0 + i + u) * steps + c];
#pragma unroll
        for (int u = 0; u < 4; ++u)
#pragma unroll
          for (int k = 0; k < kQrPanel; ++k)
            if (k < jb) cfma(w[k], cconj(Vp[(i + u) * ldv + k]), q[u]);
      }
      for (; i < mr; ++i) {
        const cplx<T> q = Q[static_cast<int64_t>(j0 + i) * steps + c];
#pragma unroll
        for (int k = 0; k < kQrPanel; ++k)
          if (k < jb) cfma(w[k], cconj(Vp[i * ldv + k]), q);
      }
      // w <- T w in place, lowest index first: w'[a] = sum_{b>=a} T[a][b] w[b]
#pragma unroll
      for (int a = 0; a < kQrPanel; ++a) {
        if (a >= jb) continue;
        cplx<T> acc = cmake<T>(0, 0);
#pragma unroll
        for (int b = a; b < kQrPanel; ++b)
          if (b < jb) cfma(acc, Tm[a * nb + b], w[b]);
        w[a] = acc;
      }
      for (int i = 0; i < mr; ++i) {
        cplx<T> &qref = Q[static_cast<int64_t>(j0 + i) * steps + c];
        cplx<T> acc = qref;
#pragma unroll
        for (int k = 0; k < kQrPanel; ++k)
          if (k < jb) {
            const cplx<T> t = cmul(Vp[i * ldv + k], w[k]);
            acc = cmake<T>(acc.re - t.re, acc.im - t.im);
          }
        qref = acc;
      }
    }
    __syncthreads();
  }
}

// One-sided (Hestenes) Jacobi SVD.  Columns of C (m x n, column-major,
// leading dimension m) are rotated pairwise until mutually orthogonal, so
// that C V = U diag(sigma); V (column-major) accumulates the rotations unless
// it is null (then only the rotated columns, U diag(sigma), are wanted).
// Round-robin ordering, one warp per column pair, the pairs of a round are
// disjoint.  A pair is left alone when its columns are orthogonal to the
// rounding level of their dot products, or when one column is negligible
// (norm at the rounding level of ||C||: no information, and its dot products
// would underflow).

// One sweep over all column pairs of C (ldc = m) with V (n x n, ld = ldv).
// Sets *flag when a rotation happened.  CTA-wide.
template <typename T>
static __device__ void onesided_sweep(int m, int n, cplx<T> *C, cplx<T> *V, int ldv, T tol, T negligible,
                               int *flag) {
  const int mm = n + (n & 1);
  const int half = mm / 2;
  for (int round = 0; round < mm - 1; ++round) {
    for (int pi = warp_id(); pi < half; pi += kWarps) {
      int p, q;
      if (pi == 0) { p = mm - 1; q = round; }
      else { p = (round + pi) % (mm - 1); q = (round - pi + (mm - 1)) % (mm - 1); }
      if (p > q) { int t = p; p = q; q = t; }
      if (q >= n) continue;
      cplx<T> *cp = C + static_cast<int64_t>(p) * m, *cq = C + static_cast<int64_t>(q) * m;
      T al = 0, be = 0, gr = 0, gi = 0;
      for (int i = lane_id(); i < m; i += 32) {
        cplx<T> x = cp[i], y = cq[i];
        al += cabs2(x);
        be += cabs2(y);
        gr += x.re * y.re + x.im * y.im;  // conj(x) y
        gi += x.re * y.im - x.im * y.re;
      }
      al = __shfl_sync(0xffffffffu, warp_sum(al), 0);
      be = __shfl_sync(0xffffffffu, warp_sum(be), 0);
      gr = __shfl_sync(0xffffffffu, warp_sum(gr), 0);
      gi = __shfl_sync(0xffffffffu, warp_sum(gi), 0);
      if (!(al > negligible) || !(be > negligible)) continue;
      T absg = sqrt(gr * gr + gi * gi);
      if (!(absg > tol * sqrt(al) * sqrt(be))) continue;
      T zeta = (be - al) / (T(2) * absg);
      T az = fabs(zeta);
      T t = az > T(1e10) ? T(0.5) / az : T(1) / (az + sqrt(T(1) + zeta * zeta));
      if (zeta < 0) t = -t;
      T cs = T(1) / sqrt(T(1) + t * t), sn = t * cs;
      cplx<T> uc = cmake<T>(gr / absg, -gi / absg);  // conj(gamma / |gamma|)
      for (int i = lane_id(); i < m; i += 32) {
        cplx<T> x = cp[i], y = cmul(uc, cq[i]);
        cp[i] = cmake<T>(cs * x.re - sn * y.re, cs * x.im - sn * y.im);
        cq[i] = cmake<T>(sn * x.re + cs * y.re, sn * x.im + cs * y.im);
      }
      if (V == nullptr) {
        if (lane_id() == 0) *flag = 1;
        continue;
      }
      cplx<T> *vp = V + static_cast<int64_t>(p) * ldv, *vq = V + static_cast<int64_t>(q) * ldv;
      for (int i = lane_id(); i < n; i += 32) {
        cplx<T> x = vp[i], y = cmul(uc, vq[i]);
        vp[i] = cmake<T>(cs * x.re - sn * y.re, cs * x.im - sn * y.im);
        vq[i] = cmake<T>(sn * x.re + cs * y.re, sn * x.im + cs * y.im);
      }
      if (lane_id() == 0) *flag = 1;
    }
    __syncthreads();
  }
}

template <typename T>
__device__ __forceinline__ T onesided_tol(int m) {
  return Eps<T>::v * T(4) * sqrt(static_cast<T>(m > 1 ? m : 1));
}

template <typename T>
static __device__ T onesided_prologue(int m, int n, const cplx<T> *C, cplx<T> *V, double *red) {
  for (int e = tid(); V != nullptr && e < n * n; e += kThreads) {
    int j = e / n, i = e % n;
    V[e] = cmake<T>(i == j ? T(1) : T(0), 0);
  }
  double fro2 = 0;
  for (int64_t e = tid(); e < static_cast<int64_t>(m) * n; e += kThreads) fro2 += cabs2d(C[e]);
  fro2 = block_sum(fro2, red);
  return static_cast<T>(static_cast<double>(Eps<T>::v) * static_cast<double>(Eps<T>::v) * fro2);
}

template <typename T, bool CL = false>
static __device__ void onesided_epilogue(int m, int n, const cplx<T> *C, T *sig2) {
  for (int j = warp_id() + kWarps * share_rank<CL>(); j < n; j += kWarps * share_size<CL>()) {
    double a = 0;
    for (int i = lane_id(); i < m; i += 32) a += cabs2d(C[static_cast<int64_t>(j) * m + i]);
    a = warp_sum(a);
    if (lane_id() == 0) sig2[j] = static_cast<T>(a);
  }
  share_sync<CL>();
}

constexpr int kMaxBlockedSweepsF = 30, kMaxBlockedSweepsD = 40;


// Unblocked: C and V wherever they are (shared memory for small problems).
template <typename T>
static __device__ __noinline__ int svd_onesided(int m, int n, cplx<T> *C, cplx<T> *V, T *sig2, int *flag, double *red) {
  const T negligible = onesided_prologue<T>(m, n, C, V, red);
  const T tol = onesided_tol<T>(m);
  const int max_sweeps = sizeof(T) == 4 ? kMaxSweepsF : kMaxSweepsD;
  int sweeps = 0;
  for (int sweep = 0; sweep < max_sweeps && n > 1; ++sweep) {
    ++sweeps;
    if (tid() == 0) *flag = 0;
    __syncthreads();
    onesided_sweep<T>(m, n, C, V, n, tol, negligible, flag);
    int f = *flag;
    __syncthreads();
    if (!f) break;
  }
  onesided_epilogue<T>(m, n, C, sig2);
  return sweeps;
}

// Blocked, for problems larger than shared memory: C (m x n, column-major)
// and V (n x n, or null) stay in global memory and the columns are split into
// blocks of bw.  One outer sweep first orthogonalises the columns inside every
// block, then lets every pair of blocks exchange its cross pairs: the block
// pairs of a tournament round are disjoint, and inside a block pair (I, J)
// step t rotates the disjoint column pairs (b, (b + t) mod w_a) over the
// smaller block's columns b and the larger block's columns, so each cross
// pair is visited once per sweep.  A visited block (or block pair) is staged
// in shared memory with its squared column norms, which a rotation updates by
// what it moves between them, so testing a pair costs one dot product.  With V, a w x w unitary Q accumulates the rotations of the visit
// and is applied to V's matching columns afterwards, a chunk of V's rows at a
// time through shared memory.  Outer sweeps repeat until one has only small rotations.
// Sum over the 16 lanes of a half warp (mask: those lanes), the same value
// broadcast to all of them.
template <typename T>
__device__ __forceinline__ T half_sum(T v, unsigned mask) {
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(mask, v, o, 16);
  return __shfl_sync(mask, v, 0, 16);
}

// One column pair (p, q) of a staged block, rotated by half a warp (the two
// halves of a warp work on two disjoint pairs).
template <typename T>
static __device__ void jacobi_rotate_staged(int m, int w, cplx<T> *Cb, cplx<T> *Q, T *nr, int p, int q, T tol,
                                     T negligible, float near, int *flag, int *any) {
  const T al = nr[p], be = nr[q];
  if (!(al > negligible) || !(be > negligible)) return;
  const int hl = lane_id() & 15;
  const unsigned mask = 0xFFFFu << (lane_id() & 16);
  cplx<T> *cp = Cb + static_cast<int64_t>(p) * m, *cq = Cb + static_cast<int64_t>(q) * m;
  T g0 = 0, g1 = 0, h0 = 0, h1 = 0;  // conj(x) y, two sums a part
  for (int i = hl; i < m; i += 16) {
    cplx<T> x = cp[i], y = cq[i];
    g0 = fma(x.re, y.re, g0);
    g1 = fma(x.im, y.im, g1);
    h0 = fma(x.re, y.im, h0);
    h1 = fma(-x.im, y.re, h1);
  }
  const T gr = half_sum(g0 + g1, mask), gi = half_sum(h0 + h1, mask);
  T cs, sn, tg;
  cplx<T> uc;
  float reach;
  if constexpr (sizeof(T) == 8) {
    // angle in single precision: the roots and divisions were 150 operations of 64 cycles
    Rotation<double> r;
    if (!make_rotation(al, be, cmake<double>(gr, gi), static_cast<float>(tol), r)) return;
    cs = r.cs;
    sn = r.sn;
    tg = r.tg;
    uc = r.uc;
    reach = r.reach;
  } else {
    const T absg = sqrt(gr * gr + gi * gi), root = sqrt(al) * sqrt(be);
    if (!(absg > tol * root)) return;
    const T zeta = (be - al) / (T(2) * absg);
    const T az = fabs(zeta);
    T t = az > T(1e10) ? T(0.5) / az : T(1) / (az + sqrt(T(1) + zeta * zeta));
    if (zeta < 0) t = -t;
    cs = T(1) / sqrt(T(1) + t * t);
    sn = t * cs;
    tg = t * absg;
    reach = fabs(t) * max(al, be) / root;
    uc = cmake<T>(gr / absg, -gi / absg);  // conj(gamma / |gamma|)
  }
  for (int i = hl; i < m; i += 16) {
    cplx<T> x = cp[i], y = cmul(uc, cq[i]);
    cp[i] = cmake<T>(cs * x.re - sn * y.re, cs * x.im - sn * y.im);
    cq[i] = cmake<T>(sn * x.re + cs * y.re, sn * x.im + cs * y.im);
  }
  if (Q != nullptr) {
    cplx<T> *qp = Q + static_cast<int64_t>(p) * w, *qq = Q + static_cast<int64_t>(q) * w;
    for (int i = hl; i < w; i += 16) {
      cplx<T> x = qp[i], y = cmul(uc, qq[i]);
      qp[i] = cmake<T>(cs * x.re - sn * y.re, cs * x.im - sn * y.im);
      qq[i] = cmake<T>(sn * x.re + cs * y.re, sn * x.im + cs * y.im);
    }
  }
  __syncwarp(mask);
  if (hl == 0) {
    nr[p] = max(al - tg, T(0));
    nr[q] = max(be + tg, T(0));
    *flag = 1;
    if (reach > near) *any = 1;
  }
}

// ---------------------------------------------------------------------------
// Register-resident cross visit of the blocked Jacobi SVD (complex64, no V).
// The two column blocks I and J (16 columns each, the last one possibly
// shorter and zero-padded) of C (m x n, column-major, m <= 256 R) are held in
// registers, thread t owning rows t, t + 256, ... of all 32 columns.  Step s
// (s = 0..15) rotates the 16 disjoint cross pairs (I_b, J_{(b+s) mod 16}):
// every thread forms its rows' contributions to the 16 complex dot products,
// one CTA-wide reduction sums them, 16 threads turn them into rotations
// (the same Hestenes rotation as onesided_sweep), and every thread applies
// them to its rows.  The J registers are then shifted by one slot, so the
// pairing stays slot b with slot b and all register indices are static.
// Column norms are reduced once per visit and then updated with the exact
// one-sided Jacobi identities |x'|^2 = |x|^2 - t|g|, |y'|^2 = |y|^2 + t|g|.
// Each column is read and written once per visit, instead of twice per pair.
// wrk: 8 * 32 + 64 + 32 floats of shared memory.  Returns whether any pair
// rotated (the columns are written back only then).

// Reduce-scatter of 32 values over a warp: lane l returns the warp sum of v[l].
__device__ __forceinline__ float warp_reduce_scatter32(float (&v)[32]) {
  const int lane = lane_id();
#pragma unroll
  for (int h = 16; h >= 1; h >>= 1) {
    const bool upper = (lane & h) != 0;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const float a = v[i], b = v[i + h];
      const float send = upper ? a : b;
      const float keep = upper ? b : a;
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, h);
    }
  }
  return v[0];
}

// CTA sum of 32 values per thread: thread i < 32 returns the sum of value i.
// Contains one barrier; red holds kWarps * 32 floats.
__device__ __forceinline__ float cta_reduce32(float (&v)[32], float *red) {
  const float s = warp_reduce_scatter32(v);
  red[warp_id() * 32 + lane_id()] = s;
  __syncthreads();
  float tot = 0.f;
  if (tid() < 32) {
#pragma unroll
    for (int w = 0; w < kWarps; ++w) tot += red[w * 32 + tid()];
  }
  return tot;
}

constexpr int kRvWrkFloats = kWarps * 32 + 64 + 32 + 4;
// sorted eigenvalues of a bond (at most 512) and, during an SVD, the
// register-visit reductions
constexpr int kLamElems = kRvWrkFloats > 512 ? kRvWrkFloats : 512;

template <int R>
static __device__ bool cross_visit_regs(int m, cplx<float> *C, int c0, int wI, int c1, int wJ, float tol,
                                        float negligible, float near, float *wrk, int *any) {
  float *red = wrk;                   // kWarps * 32
  float4 *prm = reinterpret_cast<float4 *>(wrk + kWarps * 32);  // 16 rotations
  float *nrm = wrk + kWarps * 32 + 64;  // 32 column norms: I then J (in J's column order)
  int *rot = reinterpret_cast<int *>(nrm + 32);
  cplx<float> xi[R][16], xj[R][16];
  const int t = tid();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int row = t + r * kThreads;
#pragma unroll
    for (int b = 0; b < 16; ++b) {
      xi[r][b] = (row < m && b < wI) ? C[static_cast<int64_t>(c0 + b) * m + row] : cmake<float>(0.f, 0.f);
      xj[r][b] = (row < m && b < wJ) ? C[static_cast<int64_t>(c1 + b) * m + row] : cmake<float>(0.f, 0.f);
    }
  }
  {
    float v[32];
#pragma unroll
    for (int b = 0; b < 16; ++b) {
      float a = 0.f, c = 0.f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        a += cabs2(xi[r][b]);
        c += cabs2(xj[r][b]);
      }
      v[b] = a;
      v[16 + b] = c;
    }
    const float s = cta_reduce32(v, red);
    if (t < 32) nrm[t] = s;
    if (t == 0) *rot = 0;
  }
  __syncthreads();
  for (int step = 0; step < 16; ++step) {
    float v[32];
#pragma unroll
    for (int b = 0; b < 16; ++b) {
      float gr = 0.f, gi = 0.f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const cplx<float> x = xi[r][b], y = xj[r][b];
        gr += x.re * y.re + x.im * y.im;  // conj(x) y
        gi += x.re * y.im - x.im * y.re;
      }
      v[2 * b] = gr;
      v[2 * b + 1] = gi;
    }
    const float s = cta_reduce32(v, red);
    if (t < 32) {
      const float gi = __shfl_down_sync(0xffffffffu, s, 1);
      if ((t & 1) == 0) {
        const int b = t >> 1, jb = (b + step) & 15;
        const float gr = s, al = nrm[b], be = nrm[16 + jb];
        float4 p = make_float4(1.f, 0.f, 1.f, 0.f);  // identity: skipped
        if (al > negligible && be > negligible) {
          const float absg = sqrtf(gr * gr + gi * gi), root = sqrtf(al) * sqrtf(be);
          if (absg > tol * root) {
            const float zeta = (be - al) / (2.f * absg);
            const float az = fabsf(zeta);
            float tt = az > 1e10f ? 0.5f / az : 1.f / (az + sqrtf(1.f + zeta * zeta));
            if (zeta < 0.f) tt = -tt;
            const float cs = 1.f / sqrtf(1.f + tt * tt), sn = tt * cs;
            p = make_float4(cs, sn, gr / absg, -gi / absg);  // conj(g / |g|)
            nrm[b] = fmaxf(al - tt * absg, 0.f);
            nrm[16 + jb] = fmaxf(be + tt * absg, 0.f);
            *rot = 1;
            if (fabsf(tt) * fmaxf(al, be) > near * root) *any = 1;
          }
        }
        prm[b] = p;
      }
    }
    __syncthreads();
#pragma unroll
    for (int b = 0; b < 16; ++b) {
      const float4 p = prm[b];
      if (p.x != 1.f || p.y != 0.f || p.z != 1.f || p.w != 0.f) {  // uniform over the CTA
        const cplx<float> uc = cmake<float>(p.z, p.w);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const cplx<float> x = xi[r][b], y = cmul(uc, xj[r][b]);
          xi[r][b] = cmake<float>(p.x * x.re - p.y * y.re, p.x * x.im - p.y * y.im);
          xj[r][b] = cmake<float>(p.y * x.re + p.x * y.re, p.y * x.im + p.x * y.im);
        }
      }
    }
    // slot b of J now pairs with I_b at the next step: shift J by one slot
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const cplx<float> first = xj[r][0];
#pragma unroll
      for (int b = 0; b < 15; ++b) xj[r][b] = xj[r][b + 1];
      xj[r][15] = first;
    }
  }
  __syncthreads();
  const bool rotated = *rot != 0;
  if (rotated) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int row = t + r * kThreads;
      if (row >= m) continue;
#pragma unroll
      for (int b = 0; b < 16; ++b) {
        if (b < wI) C[static_cast<int64_t>(c0 + b) * m + row] = xi[r][b];
        if (b < wJ) C[static_cast<int64_t>(c1 + b) * m + row] = xj[r][b];
      }
    }
  }
  __syncthreads();
  return rotated;
}

template <typename T>
static __device__ bool cross_visit_dispatch(int m, cplx<T> *C, int c0, int wI, int c1, int wJ, T tol, T negligible,
                                            float near, float *wrk, int *any) {
  if constexpr (sizeof(T) == 4) {
    return cross_visit_regs<1>(m, C, c0, wI, c1, wJ, tol, negligible, near, wrk, any);  // m <= kThreads
  } else {
    return false;
  }
}

// rv_wrk (kRvWrkFloats floats of shared memory, or null): with it, a
// complex64 problem without V and with m <= kThreads visits block pairs
// with cross_visit_regs (blocks of 16 columns); the blocks alone are still
// staged in shared memory.
//
// Over a cluster (CL, without V) the blocks, and then the disjoint block pairs of a
// round, go to its CTAs in turn; the stamps live in the first one's shared memory,
// read and written in place.  The arithmetic is that of one CTA.
template <typename T, bool CL = false>
static __device__ __noinline__ int svd_onesided_blocked(int m, int n, cplx<T> *C, cplx<T> *V, T *sig2, int *flag,
                                     double *red, cplx<T> *sbuf, int sbuf_elems, float *rv_wrk = nullptr) {
  const T negligible = onesided_prologue<T>(m, n, C, V, red);
  const T tol = onesided_tol<T>(m);
  // A sweep whose rotations all reach no further than `near` is the last one: what it
  // leaves is within tol (svd_small explains the bound), and the sweep that would
  // find nothing was one of 4.5.
  const float near = sqrtf(static_cast<float>(tol) / (2.5f * static_cast<float>(n)));
  // staged block pair: Q (w x w, only with V), norms (w complex slots),
  // columns (m x w)
  const bool withV = V != nullptr;
  const bool regs = sizeof(T) == 4 && !withV && rv_wrk != nullptr && m <= kThreads &&
                    static_cast<int64_t>(m) * 16 + 32 <= sbuf_elems;
  int bw = 32;
  while (bw > 1 && static_cast<int64_t>(m) * 2 * bw + (withV ? 4 * bw * bw : 0) + 2 * bw > sbuf_elems) --bw;
  if (bw > 2 * kWarps) bw -= bw % (2 * kWarps);  // whole waves of half warps per step
  if (regs) bw = 16;
  else if (CL) bw = min(bw, max(4, (n + 2 * share_size<CL>() - 1) / (2 * share_size<CL>())));  // a pair per CTA
  const int nb = (n + bw - 1) / bw, nbe = nb + (nb & 1);
  const int max_sweeps = sizeof(T) == 4 ? kMaxBlockedSweepsF : kMaxBlockedSweepsD;
  int *any = flag + 1;
  // Visits follow a fixed order (each block alone, then the tournament), so
  // visit v of sweep s has the stamp s * per_sweep + v.  last_mod[I] is the
  // stamp of the last visit that rotated columns of block I.  A visit whose
  // previous occurrence (one sweep earlier) rotated nothing, with neither
  // block changed since, would see the same columns and rotate nothing again:
  // it is skipped, which changes no result.  The stamps live in `red`, free
  // between the prologue and the epilogue.
  const int per_sweep = nb + (nbe - 1) * (nbe / 2);
  int *last_mod = reinterpret_cast<int *>(red);
  const bool skipping = nb <= static_cast<int>(kRedDoubles * sizeof(double) / sizeof(int));
  if (skipping) {
    for (int i = tid(); i < nb; i += kThreads) last_mod[i] = -1;
    share_sync<CL>();
  }
  const int ranks = share_size<CL>(), rank = share_rank<CL>();
  auto mark = [&](int I, int J, int stamp) {  // thread 0
    share_store<CL>(&last_mod[I], 0, stamp);
    share_store<CL>(&last_mod[J], 0, stamp);
  };

  auto visit = [&](int I, int J, int stamp) {
    if (skipping && stamp >= per_sweep && share_load<CL>(&last_mod[I], 0) < stamp - per_sweep &&
        share_load<CL>(&last_mod[J], 0) < stamp - per_sweep)
      return;
    const bool self = I == J;
    const int c0 = I * bw, wI = min(bw, n - c0);
    const int c1 = J * bw, wJ = self ? 0 : min(bw, n - c1);
    const int w = wI + wJ;
    if (regs && !self) {
      if (cross_visit_dispatch<T>(m, C, c0, wI, c1, wJ, tol, negligible, near, rv_wrk, any)) {
        if (skipping && tid() == 0) mark(I, J, stamp);
      }
      __syncthreads();
      return;
    }
    auto gcol = [&](int c) { return c < wI ? c0 + c : c1 + (c - wI); };
    const int qe = withV ? w * w : 0;
    cplx<T> *Q = withV ? sbuf : nullptr;
    T *nr = reinterpret_cast<T *>(sbuf + qe);
    cplx<T> *Cb = sbuf + qe + w;
    for (int e = tid(); e < m * w; e += kThreads) {
      const int c = e / m, i = e % m;
      Cb[e] = C[static_cast<int64_t>(gcol(c)) * m + i];
    }
    for (int e = tid(); e < qe; e += kThreads) Q[e] = cmake<T>((e / w) == (e % w) ? T(1) : T(0), 0);
    __syncthreads();
    for (int c = warp_id(); c < w; c += kWarps) {
      T a = 0;
      for (int i = lane_id(); i < m; i += 32) a += cabs2(Cb[static_cast<int64_t>(c) * m + i]);
      a = __shfl_sync(0xffffffffu, warp_sum(a), 0);
      if (lane_id() == 0) nr[c] = a;
    }
    if (tid() == 0) *flag = 0;
    __syncthreads();
    if (self) {
      const int mm = w + (w & 1), half = mm / 2;
      const int hw = 2 * warp_id() + (lane_id() >> 4);  // half-warp index
      for (int round = 0; round < mm - 1; ++round) {
        for (int pi = hw; pi < half; pi += 2 * kWarps) {
          int p, q;
          if (pi == 0) { p = mm - 1; q = round; }
          else { p = (round + pi) % (mm - 1); q = (round - pi + (mm - 1)) % (mm - 1); }
          if (p > q) { int tt = p; p = q; q = tt; }
          if (q >= w) continue;
          jacobi_rotate_staged<T>(m, w, Cb, Q, nr, p, q, tol, negligible, near, flag, any);
        }
        __syncthreads();
      }
    } else {
      const bool i_larger = wI >= wJ;
      const int wa = i_larger ? wI : wJ, wb = i_larger ? wJ : wI;
      const int hw = 2 * warp_id() + (lane_id() >> 4);  // half-warp index
      for (int t = 0; t < wa; ++t) {
        for (int b = hw; b < wb; b += 2 * kWarps) {
          const int a = (b + t) % wa;
          const int p = i_larger ? a : b, q = wI + (i_larger ? b : a);
          jacobi_rotate_staged<T>(m, w, Cb, Q, nr, p, q, tol, negligible, near, flag, any);
        }
        __syncthreads();
      }
    }
    const int rotated = *flag;
    __syncthreads();
    if (!rotated) return;
    if (skipping && tid() == 0) mark(I, J, stamp);
    for (int e = tid(); e < m * w; e += kThreads) {
      const int c = e / m, i = e % m;
      C[static_cast<int64_t>(gcol(c)) * m + i] = Cb[e];
    }
    __syncthreads();
    // V[:, cols] <- V[:, cols] Q, rows staged in the column buffer
    const int rows_cap = (sbuf_elems - qe - w) / w;
    for (int i0 = 0; withV && i0 < n; i0 += rows_cap) {
      const int rows = min(rows_cap, n - i0);
      for (int e = tid(); e < rows * w; e += kThreads) {
        const int c = e / rows, i = e % rows;
        Cb[e] = V[static_cast<int64_t>(gcol(c)) * n + i0 + i];
      }
      __syncthreads();
      // four output columns per thread: one staged element feeds four FMAs
      const int groups = (w + 3) / 4;
      for (int e = tid(); e < rows * groups; e += kThreads) {
        const int g = e / rows, i = e % rows, cb = 4 * g;
        cplx<T> acc[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) acc[u] = cmake<T>(0, 0);
        for (int j = 0; j < w; ++j) {
          const cplx<T> v = Cb[j * rows + i];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (cb + u < w) cfma(acc[u], v, Q[(cb + u) * w + j]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (cb + u < w) V[static_cast<int64_t>(gcol(cb + u)) * n + i0 + i] = acc[u];
      }
      __syncthreads();
    }
  };

  int sweeps = 0;
  for (int sweep = 0; sweep < max_sweeps && n > 1; ++sweep) {
    ++sweeps;
    if (tid() == 0) *any = 0;
    __syncthreads();
    const int base = sweep * per_sweep;
    for (int I = rank; I < nb; I += ranks) visit(I, I, base + I);
    if (CL) share_sync<CL>();
    for (int round = 0; round < nbe - 1; ++round) {
      for (int bp = rank; bp < nbe / 2; bp += ranks) {
        int I, J;
        if (bp == 0) { I = nbe - 1; J = round; }
        else { I = (round + bp) % (nbe - 1); J = (round - bp + (nbe - 1)) % (nbe - 1); }
        if (I > J) { int tt = I; I = J; J = tt; }
        if (J >= nb) continue;
        visit(I, J, base + nb + round * (nbe / 2) + bp);
      }
      if (CL) share_sync<CL>();
    }
    share_sync<CL>();
    int f = 0;
    for (int r = 0; r < ranks; ++r) f |= share_load<CL>(any, r);
    share_sync<CL>();
    if (!f) break;
  }
  onesided_epilogue<T, CL>(m, n, C, sig2);
  return sweeps;
}

// One Newton-Schulz step X <- X (3 I - X^dag X) / 2 on the k orthonormal-to-
// rounding columns of X (n x k, row-major, ld k): the accumulated rotations
// leave X orthonormal only to about sqrt(#rotations) eps; this brings it back
// to the rounding level of one product.  G and Y are k x k and n x k scratch.
template <typename T>
static __device__ __noinline__ void reorthonormalize(int n, int k, cplx<T> *X, cplx<T> *G, cplx<T> *Y, cplx<T> *tile) {
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  cgemm<T, 1, 0>(k, k, n, one, X, k, X, k, zero, G, k, tile);
  for (int e = tid(); e < k * k; e += kThreads) {
    int i = e / k, j = e % k;
    cplx<T> g = G[e];
    G[e] = cmake<T>((i == j ? T(1.5) : T(0)) - T(0.5) * g.re, -T(0.5) * g.im);
  }
  __syncthreads();
  cgemm<T, 0, 0>(n, k, k, one, X, k, G, k, zero, Y, k, tile);
  for (int e = tid(); e < n * k; e += kThreads) X[e] = Y[e];
  __syncthreads();
}

// Descending order of lambda (ties by index): perm[rank] = index.
template <typename T>
static __device__ void sort_desc(int n, const T *lam, int *perm) {
  for (int i = tid(); i < n; i += kThreads) perm[i] = i;
  __syncthreads();
  for (int i = tid(); i < n; i += kThreads) {
    T li = lam[i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      T lj = lam[j];
      rank += (lj > li) || (lj == li && j < i);
    }
    if (li == li && rank < n) perm[rank] = i;  // a NaN keeps the identity slot
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------
// The MPO of one rotation or measurement.
// MPO_ADJ_B: the adjoint of a case-B measurement, U |v><0|_j (U the
// controlled-Pauli product of the measurement, |v> its site-j eigenvector).
enum MpoKind { MPO_ROT = 0, MPO_PROJ_Z = 1, MPO_PROJ_B = 2, MPO_ADJ_B = 3 };

template <typename T>
struct MpoSpec {
  int kind, lo, hi, j;
  int par;         // case A: parity of the Z support that the projector keeps
  cplx<T> w0, w1;  // branch weights (folded into site lo)
  cplx<T> v0, v1;  // measurement eigenvector at site j (case B)
};

// 2x2 operator (row-major op[s*2 + t]) of branch `br` at site k of the span.
template <typename T>
static __device__ void site_op(const MpoSpec<T> &sp, const uint64_t *ppx, const uint64_t *ppz, int k,
                        int br, cplx<T> op[4]) {
  const bool x = (ppx[k >> 6] >> (k & 63)) & 1, z = (ppz[k >> 6] >> (k & 63)) & 1;
  const cplx<T> zero = cmake<T>(0, 0), one = cmake<T>(1, 0);
  op[0] = one; op[1] = zero; op[2] = zero; op[3] = one;
  if (br == 1) {
    if (sp.kind == MPO_PROJ_B && k == sp.j) {
      op[0] = zero; op[1] = cconj(sp.v1); op[2] = zero; op[3] = zero;
    } else if (sp.kind == MPO_ADJ_B && k == sp.j) {  // v1 |1><0|
      op[0] = zero; op[1] = zero; op[2] = sp.v1; op[3] = zero;
    } else if (sp.kind == MPO_PROJ_B || sp.kind == MPO_ADJ_B) {
      // Hermitian letter of P' at k (controlled-Pauli target)
      if (x && !z) { op[0] = zero; op[1] = one; op[2] = one; op[3] = zero; }
      else if (x && z) { op[0] = zero; op[1] = cmake<T>(0, -1); op[2] = cmake<T>(0, 1); op[3] = zero; }
      else if (z) { op[3] = cmake<T>(-1, 0); }
    } else {
      // X^x Z^z (MPO_PROJ_Z has x = 0 on every site)
      if (x && !z) { op[0] = zero; op[1] = one; op[2] = one; op[3] = zero; }
      else if (x && z) { op[0] = zero; op[1] = cmake<T>(-1, 0); op[2] = one; op[3] = zero; }
      else if (z) { op[3] = cmake<T>(-1, 0); }
    }
  } else if (sp.kind == MPO_PROJ_B && k == sp.j) {
    op[0] = cconj(sp.v0); op[3] = zero;
  } else if (sp.kind == MPO_ADJ_B && k == sp.j) {  // v0 |0><0|
    op[0] = sp.v0; op[3] = zero;
  }
  if (k == sp.lo) {
    cplx<T> w = br == 0 ? sp.w0 : sp.w1;
    for (int i = 0; i < 4; ++i) op[i] = cmul(w, op[i]);
  }
}

// ---------------------------------------------------------------------------
// Shared-memory layout of the round kernel.
template <typename T>
struct Smem {
  uint64_t *tx, *tz, *ppx, *ppz;
  uint8_t *tm;
  int *chi, *perm, *misc;
  int64_t *off;  // span offsets: Ap stack [n+2], G stack [n+2]
  int64_t *goff;
  double *red;
  double *dmisc;
  cplx<T> *tile;
  cplx<T> *jbuf;
  int *rdim;
  T *lam;
  MpoSpec<T> *spec;
};

template <typename T>
__host__ __device__ size_t smem_bytes(int n, int W, int svd_elems) {
  size_t b = 0;
  auto add = [&](size_t bytes) { b += (bytes + 15) & ~size_t(15); };
  add(sizeof(uint64_t) * 2 * n * W);  // tx
  add(sizeof(uint64_t) * 2 * n * W);  // tz
  add(sizeof(uint64_t) * W);          // ppx
  add(sizeof(uint64_t) * W);          // ppz
  add(2 * n);                         // tm
  add(sizeof(int) * (n + 2));         // chi
  add(sizeof(int) * 512);             // perm
  add(sizeof(int) * 16);              // misc
  add(sizeof(int64_t) * (n + 2));     // off
  add(sizeof(int64_t) * (n + 2));     // goff
  add(sizeof(double) * kRedDoubles);  // red
  add(sizeof(double) * 24);           // dmisc
  if (!kLight) add(sizeof(cplx<T>) * kTileElems);  // tile
  add(sizeof(cplx<T>) * svd_elems);  // jbuf
  add(sizeof(int) * (n + 2));         // rdim
  add(sizeof(T) * kLamElems);         // lam (also the register-visit reductions)
  add(sizeof(MpoSpec<T>));
  return b;
}

// Largest SVD buffer (complex elements, at most SvdSmem) that keeps the round
// kernel within the 227 KB of shared memory a CTA may use, or two CTAs within
// the 228 KB of an SM (1 KB of which each CTA reserves).
template <typename T>
inline int svd_elems_for(int n, int W) {
  const size_t limit = (kLight ? 112 : 227) * 1024;
  const size_t base = smem_bytes<T>(n, W, 0);
  if (base + 64 >= limit) return 0;
  const size_t e = (limit - base - 64) / sizeof(cplx<T>);
  return static_cast<int>(e < static_cast<size_t>(SvdSmem<T>::elems) ? e : SvdSmem<T>::elems);
}

template <typename T>
static __device__ Smem<T> carve(char *base, int n, int W, int svd_elems) {
  Smem<T> s;
  size_t b = 0;
  auto take = [&](size_t bytes) {
    char *p = base + b;
    b += (bytes + 15) & ~size_t(15);
    return p;
  };
  s.tx = reinterpret_cast<uint64_t *>(take(sizeof(uint64_t) * 2 * n * W));
  s.tz = reinterpret_cast<uint64_t *>(take(sizeof(uint64_t) * 2 * n * W));
  s.ppx = reinterpret_cast<uint64_t *>(take(sizeof(uint64_t) * W));
  s.ppz = reinterpret_cast<uint64_t *>(take(sizeof(uint64_t) * W));
  s.tm = reinterpret_cast<uint8_t *>(take(2 * n));
  s.chi = reinterpret_cast<int *>(take(sizeof(int) * (n + 2)));
  s.perm = reinterpret_cast<int *>(take(sizeof(int) * 512));
  s.misc = reinterpret_cast<int *>(take(sizeof(int) * 16));
  s.off = reinterpret_cast<int64_t *>(take(sizeof(int64_t) * (n + 2)));
  s.goff = reinterpret_cast<int64_t *>(take(sizeof(int64_t) * (n + 2)));
  s.red = reinterpret_cast<double *>(take(sizeof(double) * kRedDoubles));
  s.dmisc = reinterpret_cast<double *>(take(sizeof(double) * 24));
  if (!kLight) s.tile = reinterpret_cast<cplx<T> *>(take(sizeof(cplx<T>) * kTileElems));
  s.jbuf = reinterpret_cast<cplx<T> *>(take(sizeof(cplx<T>) * svd_elems));
  if (kLight) s.tile = s.jbuf;  // free whenever a GEMM runs
  s.rdim = reinterpret_cast<int *>(take(sizeof(int) * (n + 2)));
  s.lam = reinterpret_cast<T *>(take(sizeof(T) * kLamElems));
  s.spec = reinterpret_cast<MpoSpec<T> *>(take(sizeof(MpoSpec<T>)));
  return s;
}

// misc slots
// (M_JFLAG + 1 holds the blocked Jacobi's sweep flag; M_TICKET the shot taken from the queue)
enum { M_LO = 0, M_HI, M_A, M_B, M_CENTER, M_FAIL, M_KEEP, M_MAXCHI, M_CASEB, M_J, M_BIT, M_LIDX, M_OUTCOME, M_JFLAG,
       M_TICKET = 15 };
// dmisc slots
enum { D_DISC = 0, D_LOGP, D_E, D_NORM, D_FLOPS = 8, D_PROF = 8 };  // D_PROF + 1 + ProfSlot

// The slots from D_FLOPS on hold integers.
__device__ __forceinline__ long long &tally(double *dmisc, int slot) { return reinterpret_cast<long long *>(dmisc)[slot]; }

// Adds the cycles since `t` to a phase slot and restarts `t` (thread 0 only;
// callers sit just after a CTA barrier so the CTA is in step).
__device__ __forceinline__ void prof_mark(double *dmisc, int slot, long long &t) {
  if (threadIdx.x == 0) {
    const long long now = clock64();
    tally(dmisc, D_PROF + 1 + slot) += now - t;
    t = now;
  }
}

// Per-CTA scratch partition (complex elements).
template <typename T>
struct Scratch {
  cplx<T> *ap, *g, *t, *y, *h, *v, *vs, *w, *mbuf, *e, *sa, *te;
  T *lam;
};

template <typename T>
static __device__ Scratch<T> scratch_for(const EngineParams &P, int cap) {
  Scratch<T> s;
  cplx<T> *base = reinterpret_cast<cplx<T> *>(P.scratch) + static_cast<int64_t>(blockIdx.x) * P.scratch_elems;
  const int64_t c2 = static_cast<int64_t>(cap) * cap;
  s.ap = base;
  s.g = s.ap + P.ap_elems;
  s.t = s.g + P.g_elems;
  s.y = s.t + 8 * c2;
  s.h = s.y + 4 * c2;
  s.v = s.h + 4 * c2;
  s.vs = s.v + 4 * c2;
  s.w = s.vs + 4 * c2;
  s.mbuf = s.w + 2 * c2;
  s.e = s.mbuf + 4 * c2;
  s.sa = s.e + c2;
  s.te = s.sa + 2 * c2;
  s.lam = reinterpret_cast<T *>(s.te + 2 * c2);
  return s;
}

// Algorithmic FLOP counts (real flops of the textbook algorithm, complex = 4
// real multiply-adds per multiply-add): a GEMM is 8 M N K, a Householder R
// factor of an m x n matrix 4 (2 m n^2 - 2 n^3 / 3) with m >= n, the
// singular values and the vectors of the smaller side of an m x n matrix
// 4 (4 m n^2 + 8 n^3) with m >= n (roles swapped otherwise in both).
// An R factor counts also where the matrix is its own R and none is computed: the
// count is the algorithm's, and stays comparable.
// In thirds of a flop: thread 0 counts in integers, since a double-precision
// operation takes 64 cycles and these were 40 a bond, of about 70,000 cycles.
static __device__ __forceinline__ long long gemm_flops(int M, int N, int K) { return 24ll * M * N * K; }
static __device__ __forceinline__ long long qr_flops(int m, int n) {
  const long long a = max(m, n), b = min(m, n);
  return (24 * a - 8 * b) * b * b;
}
static __device__ __forceinline__ long long svd_flops(int m, int n) {
  const long long a = max(m, n), b = min(m, n);
  return (48 * a + 96 * b) * b * b;
}

// ---------------------------------------------------------------------------
// MPS pieces (CTA-wide).
template <typename T>
__device__ __forceinline__ cplx<T> *site_ptr(const EngineParams &P, int64_t shot, int k) {
  return reinterpret_cast<cplx<T> *>(P.mps) + shot * P.slab_elems + P.site_off[k];
}

// out = branch-summed MPO tensor of site k (see header comment): left bond
// doubled when dl, right bond doubled when dr; the (alpha, l) index is
// alpha * chl + l.  Elements first, first + stride, ... by the calling thread.
template <typename T>
static __device__ __noinline__ void materialize(const MpoSpec<T> &sp, const uint64_t *ppx, const uint64_t *ppz, int k,
                            const cplx<T> *A, int chl, int chr, bool dl, bool dr, cplx<T> *out,
                            int first, int stride) {
  if (sp.kind == MPO_PROJ_Z) {
    // (I + s Z_S)/2 written without its two cancelling branches: the bond
    // index carries the parity of the S bits to the left, a site in S adds
    // its own bit, and the last site keeps only the target parity.  All
    // entries are 0 or 1, so a small Born probability is not the difference
    // of two numbers of order one.
    const bool in_s = (ppz[k >> 6] >> (k & 63)) & 1;
    const int Dl = dl ? 2 * chl : chl, Dr = dr ? 2 * chr : chr;
    const int total = Dl * 2 * Dr;
    for (int e = first; e < total; e += stride) {
      const int R = e % Dr;
      const int sb = (e / Dr) & 1;
      const int L = e / (2 * Dr);
      const int al = dl ? L / chl : 0, l = dl ? L % chl : L;
      const int be = dr ? R / chr : sp.par, r = dr ? R % chr : R;
      const bool keep = in_s ? ((al ^ sb) == be) : (al == be);
      out[e] = keep ? A[(static_cast<int64_t>(l) * 2 + sb) * chr + r] : cmake<T>(0, 0);
    }
    return;
  }
  cplx<T> op0[4], op1[4];
  site_op(sp, ppx, ppz, k, 0, op0);
  site_op(sp, ppx, ppz, k, 1, op1);
  const int Dl = dl ? 2 * chl : chl, Dr = dr ? 2 * chr : chr;
  const int total = Dl * 2 * Dr;
  for (int e = first; e < total; e += stride) {
    int R = e % Dr;
    int s = (e / Dr) & 1;
    int L = e / (2 * Dr);
    int al = dl ? L / chl : -1, l = dl ? L % chl : L;
    int be = dr ? R / chr : -1, r = dr ? R % chr : R;
    cplx<T> val = cmake<T>(0, 0);
    if (!(dl && dr && al != be)) {
      int br = dl ? al : be;
      cplx<T> a0 = A[(static_cast<int64_t>(l) * 2 + 0) * chr + r];
      cplx<T> a1 = A[(static_cast<int64_t>(l) * 2 + 1) * chr + r];
      if (br < 0) {
        cfma(val, cadd(op0[s * 2 + 0], op1[s * 2 + 0]), a0);
        cfma(val, cadd(op0[s * 2 + 1], op1[s * 2 + 1]), a1);
      } else {
        const cplx<T> *op = br == 0 ? op0 : op1;
        cfma(val, op[s * 2 + 0], a0);
        cfma(val, op[s * 2 + 1], a1);
      }
    }
    out[e] = val;
  }
}

// Exact gauge steps (no truncation) moving the orthogonality centre of a
// shot's MPS from its current site to `target`, so that the sites left of an
// operator's support are left-canonical and those right of it
// right-canonical before the operator is applied (Sec. IV B).
//   Right across site k: A_k as a (2 chi_k) x chi_{k+1} matrix = Q R
//   (Householder); site k becomes Q (bond k+1 becomes min(2 chi_k,
//   chi_{k+1})) and A_{k+1} <- R A_{k+1}.
//   Left across site k: A_k^dag as a (2 chi_{k+1}) x chi_k matrix = Q R;
//   site k becomes Q^dag and A_{k-1} <- A_{k-1} R^dag.
// A matrix with no more rows than columns is its own R, with Q = 1.
template <typename T>
static __device__ __noinline__ void mps_move_center(const EngineParams &P, const Smem<T> &S, int64_t shot, const Scratch<T> &X,
                                int target) {
  int *chi = S.chi;
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  int c = S.misc[M_CENTER];
  while (c < target) {
    const int l = chi[c], r = chi[c + 1], r2 = chi[c + 2];
    const int m = 2 * l, steps = min(m, r);
    if (m > kMaxVec) {
      if (tid() == 0) S.misc[M_FAIL] = STN_EOVERFLOW;
      __syncthreads();
      return;
    }
    cplx<T> *A = site_ptr<T>(P, shot, c), *Bn = site_ptr<T>(P, shot, c + 1);
    if (m <= r) {
      cgemm<T, 0, 0>(m, 2 * r2, r, one, A, r, Bn, 2 * r2, zero, X.w, 2 * r2, S.tile);
      for (int e = tid(); e < m * m; e += kThreads) A[e] = cmake<T>(T(e / m == e % m), 0);
    } else if (qr_small_elems(m, r, true) <= P.svd_elems) {
      qr_small<T>(m, r, A, r, false, X.t, steps, A, S.jbuf);
      cgemm<T, 0, 0>(steps, 2 * r2, r, one, X.t, r, Bn, 2 * r2, zero, X.w, 2 * r2, S.tile);
    } else {
      for (int e = tid(); e < m * r; e += kThreads) X.t[e] = A[e];
      __syncthreads();
      qr_r_inplace<T>(m, r, X.t, r, S.jbuf, P.svd_elems, X.h);
      form_q<T>(m, steps, X.h, X.y, S.jbuf, P.svd_elems);
      cgemm<T, 0, 0>(steps, 2 * r2, r, one, X.t, r, Bn, 2 * r2, zero, X.w, 2 * r2, S.tile);
      for (int e = tid(); e < m * steps; e += kThreads) A[e] = X.y[e];
    }
    for (int e = tid(); e < steps * 2 * r2; e += kThreads) Bn[e] = X.w[e];
    if (tid() == 0) {
      chi[c + 1] = steps;
      tally(S.dmisc, D_FLOPS) += 2 * qr_flops(m, r) + gemm_flops(steps, 2 * r2, r);
      tally(S.dmisc, D_PROF + 1 + PROF_NGAUGE) += 1;
    }
    __syncthreads();
    ++c;
  }
  while (c > target) {
    const int l = chi[c], r = chi[c + 1], ll = chi[c - 1];
    const int m = 2 * r, steps = min(m, l);
    if (m > kMaxVec) {
      if (tid() == 0) S.misc[M_FAIL] = STN_EOVERFLOW;
      __syncthreads();
      return;
    }
    cplx<T> *A = site_ptr<T>(P, shot, c), *Am = site_ptr<T>(P, shot, c - 1);
    if (m <= l) {
      cgemm<T, 0, 0>(2 * ll, m, l, one, Am, l, A, m, zero, X.w, m, S.tile);
      for (int e = tid(); e < m * m; e += kThreads) A[e] = cmake<T>(T(e / m == e % m), 0);
    } else if (qr_small_elems(m, l, true) <= P.svd_elems) {
      qr_small<T>(m, l, A, m, true, X.t, steps, A, S.jbuf);
      cgemm<T, 0, 1>(2 * ll, steps, l, one, Am, l, X.t, l, zero, X.w, steps, S.tile);
    } else {
      for (int e = tid(); e < m * l; e += kThreads) {
        const int j = e / l, i = e % l;  // X.t[j][i] = conj(A[i][j]), A as l x 2r
        X.t[e] = cconj(A[static_cast<int64_t>(i) * m + j]);
      }
      __syncthreads();
      qr_r_inplace<T>(m, l, X.t, l, S.jbuf, P.svd_elems, X.h);
      form_q<T>(m, steps, X.h, X.y, S.jbuf, P.svd_elems);
      cgemm<T, 0, 1>(2 * ll, steps, l, one, Am, l, X.t, l, zero, X.w, steps, S.tile);
      for (int e = tid(); e < steps * m; e += kThreads) {
        const int k = e / m, j = e % m;
        A[e] = cconj(X.y[static_cast<int64_t>(j) * steps + k]);
      }
    }
    for (int e = tid(); e < 2 * ll * steps; e += kThreads) Am[e] = X.w[e];
    if (tid() == 0) {
      chi[c] = steps;
      tally(S.dmisc, D_FLOPS) += 2 * qr_flops(m, l) + gemm_flops(2 * ll, steps, l);
      tally(S.dmisc, D_PROF + 1 + PROF_NGAUGE) += 1;
    }
    __syncthreads();
    --c;
  }
  if (tid() == 0) S.misc[M_CENTER] = target;
  __syncthreads();
}

// Two phases of applying the two-branch MPO `spec` on [lo, hi] and
// recompressing sites [a, b] (a <= lo <= hi <= b, orthogonality centre inside
// [a, b]).
//
// mps_prepare builds the MPO tensors and runs the left sweep (no truncation
// yet) and returns the squared norm of the new, untruncated state: for a
// measurement projector this is the Born probability of the branch, obtained
// from R factors whose small entries carry absolute (not relative) rounding,
// so a small probability keeps its relative accuracy (about eps / sqrt(p)).
// mps_finish then runs the truncating right sweep; the centre ends at a and the
// state is renormalised.
template <typename T>
static __device__ __noinline__ double mps_prepare(const EngineParams &P, const Smem<T> &S, int64_t shot,
                              const Scratch<T> &X, int a, int b, bool want_norm) {
  const MpoSpec<T> &sp = *S.spec;
  int *chi = S.chi;
  if (a == b) {
    cplx<T> *A = site_ptr<T>(P, shot, a);
    materialize(sp, S.ppx, S.ppz, a, A, chi[a], chi[a + 1], false, false, X.t, tid(), kThreads);
    __syncthreads();
    if (!want_norm) return 0.0;
    const int64_t tot = static_cast<int64_t>(chi[a]) * 2 * chi[a + 1];
    double nrm = 0;
    for (int64_t e = tid(); e < tot; e += kThreads) nrm += cabs2d(X.t[e]);
    return block_sum(nrm, S.red);
  }
  // doubled bond dimensions D[k] for bonds a..b+1
  auto Dbond = [&](int k) { return (k > sp.lo && k <= sp.hi) ? 2 * chi[k] : chi[k]; };
  __syncthreads();  // the callers have read M_FAIL, which may be written here
  if (tid() == 0) {
    int64_t o = 0;
    for (int k = a; k <= b; ++k) {
      S.off[k - a] = o;
      o += static_cast<int64_t>(Dbond(k)) * 2 * Dbond(k + 1);
    }
    S.off[b - a + 1] = o;
    int64_t g = 0;
    for (int k = a + 1; k <= b; ++k) {
      S.goff[k - a] = g;
      g += static_cast<int64_t>(Dbond(k)) * Dbond(k);
    }
    S.goff[b - a + 1] = g;
    if (o > P.ap_elems || g > P.g_elems) S.misc[M_FAIL] = STN_EOVERFLOW;
  }
  __syncthreads();
  if (S.misc[M_FAIL]) return 0.0;
  // Doubled sites: one of up to kWarpSite elements by a warp, the span's sites
  // in parallel (a site's tensor is a chain of index arithmetic and two loads:
  // 5000 cycles, which the whole CTA would spend per site); a larger one by
  // the CTA.  (With 256 or 4096 elements for 1024 the workloads measured stay within 1 %.)
  // The span is the operator's support, so a <= lo <= hi <= b hold with equality.
  constexpr int kWarpSite = 1024;
  for (int pass = 0; pass < 2; ++pass) {
    for (int k = pass == 0 ? a + warp_id() : a; k <= b; k += pass == 0 ? kWarps : 1) {
      const bool dl = k > sp.lo, dr = k < sp.hi;
      const bool by_warp = Dbond(k) * 2 * Dbond(k + 1) <= kWarpSite;
      if (by_warp != (pass == 0)) continue;
      materialize(sp, S.ppx, S.ppz, k, site_ptr<T>(P, shot, k), chi[k], chi[k + 1], dl, dr, X.ap + S.off[k - a],
                  by_warp ? lane_id() : tid(), by_warp ? 32 : kThreads);
    }
  }
  __syncthreads();
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  // left sweep: R factor of the left part through site k, for k = a..b-1
  // (R at bond a is the identity: sites left of a are left-canonical).
  for (int k = a; k < b; ++k) {
    const int Dl = Dbond(k), Dr = Dbond(k + 1);
    const cplx<T> *Ak = X.ap + S.off[k - a];
    cplx<T> *Rout = X.g + S.goff[k + 1 - a];
    int m;
    const cplx<T> *src = X.t;
    // A matrix with no more rows than columns is an R as it stands (any R with the
    // same R^dag R will do): it goes where R goes.  That is the first site of most
    // spans: a d = 5 round at theta = 0.05 takes 158 ms instead of 165, two d = 3
    // rounds in complex128 54.6 instead of 59.8.
    bool is_r;
    if (k == a) {
      m = 2 * Dl;
      src = Ak;
      is_r = m <= Dr;
      if (is_r)
        for (int e = tid(); e < m * Dr; e += kThreads) Rout[e] = Ak[e];
    } else {
      const int r = S.rdim[k - a];
      const cplx<T> *Rk = X.g + S.goff[k - a];
      m = 2 * r;
      is_r = m <= Dr;
      cgemm<T, 0, 0>(r, 2 * Dr, Dl, one, Rk, Dl, Ak, 2 * Dr, zero, is_r ? Rout : X.t, 2 * Dr, S.tile);
      if (tid() == 0) tally(S.dmisc, D_FLOPS) += gemm_flops(r, 2 * Dr, Dl);
    }
    if (m > kMaxVec) {
      if (tid() == 0) S.misc[M_FAIL] = STN_EOVERFLOW;
      __syncthreads();
      return 0.0;
    }
    if (tid() == 0) tally(S.dmisc, D_FLOPS) += qr_flops(m, Dr);
    const int rn = min(m, Dr);
    if (!is_r && qr_small_elems(m, Dr, false) <= P.svd_elems) {
      qr_small<T>(m, Dr, src, Dr, false, Rout, rn, nullptr, S.jbuf);
    } else if (!is_r) {
      if (src != X.t) {
        for (int e = tid(); e < m * Dr; e += kThreads) X.t[e] = src[e];
        __syncthreads();
      }
      qr_r_inplace<T>(m, Dr, X.t, Dr, S.jbuf, P.svd_elems);
      for (int e = tid(); e < rn * Dr; e += kThreads) Rout[e] = X.t[e];
    }
    if (tid() == 0) S.rdim[k + 1 - a] = rn;
    __syncthreads();
  }
  // R_b A'_b, the first matrix of the right sweep, stays in X.y for mps_finish;
  // squared norm of the state: its Frobenius norm (the right part beyond b is
  // right-canonical)
  {
    const int Dl = Dbond(b), n2 = 2 * Dbond(b + 1), r = S.rdim[b - a];
    cgemm<T, 0, 0>(r, n2, Dl, one, X.g + S.goff[b - a], Dl, X.ap + S.off[b - a], n2, zero, X.y, n2, S.tile);
    if (!want_norm) return 0.0;
    double nrm = 0;
    for (int e = tid(); e < r * n2; e += kThreads) nrm += cabs2d(X.y[e]);
    return block_sum(nrm, S.red);
  }
}

template <typename T>
static __device__ __noinline__ void mps_finish(const EngineParams &P, const Smem<T> &S, int64_t shot, const Scratch<T> &X,
                           int a, int b) {
  const MpoSpec<T> &sp = *S.spec;
  int *chi = S.chi;
  const int cap = P.chi_cap;
  if (S.misc[M_FAIL]) return;
  if (a == b) {
    cplx<T> *A = site_ptr<T>(P, shot, a);
    const int64_t tot = static_cast<int64_t>(chi[a]) * 2 * chi[a + 1];
    double nrm = 0;
    for (int64_t e = tid(); e < tot; e += kThreads) nrm += cabs2d(X.t[e]);
    nrm = block_sum(nrm, S.red);
    T inv = static_cast<T>(nrm > 0 ? 1.0 / sqrt(nrm) : 0.0);
    for (int64_t e = tid(); e < tot; e += kThreads) A[e] = cscale(X.t[e], inv);
    if (tid() == 0) {
      if (!(nrm > 0) || !isfinite(nrm)) S.misc[M_FAIL] = STN_ENUMERIC;
      S.misc[M_CENTER] = a;
    }
    __syncthreads();
    return;
  }
  auto Dbond = [&](int k) { return (k > sp.lo && k <= sp.hi) ? 2 * chi[k] : chi[k]; };
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  long long tp = clock64();
  // right sweep
  int kappa = Dbond(b + 1);
  const cplx<T> *M = X.ap + S.off[b - a];
  for (int k = b; k > a; --k) {
    const int Dl = Dbond(k);
    const int n2 = 2 * kappa;
    const int r = S.rdim[k - a];
    const cplx<T> *Rk = X.g + S.goff[k - a];
    // C = R_k M (r x n2; mps_prepare left the first one in X.y), then its SVD
    if (k < b) cgemm<T, 0, 0>(r, n2, Dl, one, Rk, Dl, M, n2, zero, X.y, n2, S.tile);
    prof_mark(S.dmisc, PROF_RIGHT, tp);
    const bool in_smem = r * n2 + n2 * n2 <= P.svd_elems;
    cplx<T> *Cc = in_smem ? S.jbuf : X.h;
    cplx<T> *Vc = in_smem ? S.jbuf + r * n2 : X.v;
    // In the complex64 path a bond whose SVD (with V) fits shared memory in
    // 16-byte numbers is decomposed in pairs of floats: FP32 Jacobi rotations leave
    // the small singular directions with an absolute error of about
    // sqrt(#rotations) eps sigma_1, which would be dropped or kept wrongly at
    // every sweep.  In complex128, every bond of up to
    // kSmallSvdCols columns takes this path.
    bool vec_from_columns = false;
    int keep = 0;
    cplx<T> *Bk = site_ptr<T>(P, shot, k);
    const int kmax = min(cap, P.chimax[k]);
    const int dscale = static_cast<int>(sizeof(double) / sizeof(T));
    const bool svd64 = n2 <= kSmallSvdCols && r <= kMaxVec &&
                       (sizeof(T) == 8 || (!P.svd64_all && 2 * (r * n2 + n2 * n2) <= P.svd_rule));
    if (svd64) {
      const int elems = n2 * (r | 1) * dscale;
      const Truncation<T> tr{S.perm, kmax, P.delta, &S.misc[M_FAIL], &S.misc[M_KEEP], &S.dmisc[D_DISC], X.vs, Bk};
      if (elems + 3 * dscale <= P.svd_elems)
        keep = svd_small<T, true>(r, n2, X.y, nullptr, S.lam, P.cutoff, S.jbuf, S.jbuf + elems, S.red, &tr);
      else  // X.t is free in the right sweep and holds it: r n2 <= 4 c^2 numbers of 16 bytes
        keep = svd_small<T, false>(r, n2, X.y, nullptr, S.lam, P.cutoff, X.t, S.jbuf, S.red, &tr);
    } else if (sizeof(T) == 4 && P.svd64_all) {
      // Complex64 contractions with every SVD in double precision: the large
      // path (Householder R factor, Jacobi on R^dag) on a complex128 copy of
      // C in the scratch areas h and v (contiguous, 4 c^2 complex128), with
      // the shared buffer as complex128 staging; the rotated columns come back
      // in single precision.
      if (r > kMaxVec) {
        if (tid() == 0) S.misc[M_FAIL] = STN_EOVERFLOW;
        __syncthreads();
        return;
      }
      cplx<double> *Cd = reinterpret_cast<cplx<double> *>(X.h);
      cplx<double> *jd = reinterpret_cast<cplx<double> *>(S.jbuf);
      double *sd = reinterpret_cast<double *>(X.te);
      for (int e = tid(); e < r * n2; e += kThreads)
        Cd[e] = cmake<double>(static_cast<double>(X.y[e].re), static_cast<double>(X.y[e].im));
      __syncthreads();
      if (n2 <= kSmallSvdCols && 2 * (n2 * (r | 1) + 3) <= P.svd_elems) {  // a small bond: svd_small on the copy
        cplx<double> *Vd = reinterpret_cast<cplx<double> *>(X.t);  // free in the right sweep, 4 c^2 complex128
        const int cols = max(1, svd_small<double, true>(r, n2, Cd, Vd, sd, P.cutoff, jd, jd + n2 * (r | 1), S.red));
        for (int e = tid(); e < n2 * cols; e += kThreads)
          X.y[e] = cmake<T>(static_cast<T>(Vd[e].re), static_cast<T>(Vd[e].im));
        for (int i = tid(); i < n2; i += kThreads) X.lam[i] = static_cast<T>(sd[i]);
        Vc = X.y;
      } else {
        const long long tqr = clock64();
        qr_r_inplace<double>(r, n2, Cd, n2, jd, P.svd_elems / 2);
        if (tid() == 0) tally(S.dmisc, D_PROF + 1 + PROF_SVD_QR) += clock64() - tqr;
        const int kx = min(r, n2);
        for (int e = tid(); e < n2 * kx; e += kThreads) Cd[e] = cconj(Cd[e]);
        __syncthreads();
        const long long tj = clock64();
        const int sweeps = svd_onesided_blocked<double>(n2, kx, Cd, nullptr, sd, &S.misc[M_JFLAG], S.red, jd,
                                                        P.svd_elems / 2);
        if (tid() == 0) {
          tally(S.dmisc, D_PROF + 1 + PROF_JSWEEPS) += sweeps;
          tally(S.dmisc, D_PROF + 1 + PROF_JROWS) += n2;
          tally(S.dmisc, D_PROF + 1 + PROF_JCOLS) += kx;
          if (n2 <= kThreads / 2) tally(S.dmisc, D_PROF + 1 + PROF_JAC_ROWS256) += clock64() - tj;
        }
        for (int e = tid(); e < n2 * kx; e += kThreads)
          X.y[e] = cmake<T>(static_cast<T>(Cd[e].re), static_cast<T>(Cd[e].im));
        for (int i = tid(); i < n2; i += kThreads) X.lam[i] = i < kx ? static_cast<T>(sd[i]) : T(0);
        __syncthreads();
        Vc = X.y;
        vec_from_columns = true;
      }
    } else if (in_smem) {
      for (int e = tid(); e < r * n2; e += kThreads) {
        int i = e / n2, j = e % n2;
        Cc[j * r + i] = X.y[e];
      }
      __syncthreads();
      svd_onesided<T>(r, n2, Cc, Vc, X.lam, &S.misc[M_JFLAG], S.red);
    } else {
      // Large bond: C = Q1 R1 (Householder), then one-sided Jacobi on
      // X = R1^dag (n2 x kx), whose columns converge in a few sweeps because
      // R1 is already nearly diagonal.  X V_x = U_x Sigma gives
      // R1 = V_x Sigma U_x^dag, so the right singular vectors of C are the
      // normalised columns of the rotated X and no rotation is accumulated.
      // Rows of R1 (row-major, ld n2) are the conjugated columns of X
      // (column-major, ld n2) in place.
      if (r > kMaxVec) {
        if (tid() == 0) S.misc[M_FAIL] = STN_EOVERFLOW;
        __syncthreads();
        return;
      }
      const long long tqr = clock64();
      qr_r_inplace<T>(r, n2, X.y, n2, S.jbuf, P.svd_elems);
      if (tid() == 0) tally(S.dmisc, D_PROF + 1 + PROF_SVD_QR) += clock64() - tqr;
      const int kx = min(r, n2);
      // complex64 with more than one block of 16 columns: blocked Jacobi
      // with register-resident block pairs, X in global scratch (L2)
      const bool regs = sizeof(T) == 4 && kx > 16 && n2 <= kThreads;
      const bool x_smem = !regs && n2 * kx <= P.svd_elems;
      cplx<T> *Xc = x_smem ? S.jbuf : X.y;
      for (int e = tid(); e < n2 * kx; e += kThreads) Xc[e] = cconj(X.y[e]);
      __syncthreads();
      const long long tj = clock64();
      const int sweeps =
          x_smem ? svd_onesided<T>(n2, kx, Xc, nullptr, X.lam, &S.misc[M_JFLAG], S.red)
                 : svd_onesided_blocked<T>(n2, kx, Xc, nullptr, X.lam, &S.misc[M_JFLAG], S.red, S.jbuf,
                                           P.svd_elems, regs ? reinterpret_cast<float *>(S.lam) : nullptr);
      if (tid() == 0) {
        tally(S.dmisc, D_PROF + 1 + PROF_JSWEEPS) += sweeps;
        tally(S.dmisc, D_PROF + 1 + PROF_JROWS) += n2;
        tally(S.dmisc, D_PROF + 1 + PROF_JCOLS) += kx;
        if (n2 <= kThreads / 2) tally(S.dmisc, D_PROF + 1 + PROF_JAC_ROWS256) += clock64() - tj;
      }
      for (int i = kx + tid(); i < n2; i += kThreads) X.lam[i] = T(0);
      __syncthreads();
      Vc = Xc;
      vec_from_columns = true;
    }
    __syncthreads();
    if (tid() == 0 && !vec_from_columns) tally(S.dmisc, D_PROF + 1 + PROF_SVD_SMALL) += clock64() - tp;
    prof_mark(S.dmisc, PROF_SVD, tp);
    if (tid() == 0) {
      tally(S.dmisc, D_FLOPS) += gemm_flops(r, n2, Dl) + svd_flops(r, n2);
      tally(S.dmisc, D_PROF + 1 + (vec_from_columns ? PROF_NSVD_LARGE : PROF_NSVD_SMALL)) += 1;
    }
    const bool rounded = sizeof(T) == 4 && !vec_from_columns && (svd64 || P.svd64_all);
    if (svd64) {
      if (S.misc[M_FAIL]) return;
    } else {  // no thread reads M_FAIL here before the barrier that follows its write
      // S.lam holds the squared values, S.perm their order
      for (int i = tid(); i < n2; i += kThreads) {
        const T l = X.lam[i];
        const bool bad = !isfinite(l);
        if (bad) S.misc[M_FAIL] = STN_ENUMERIC;
        S.lam[i] = bad ? T(0) : l;
      }
      __syncthreads();
      if (S.misc[M_FAIL]) return;
      sort_desc<T>(n2, S.lam, S.perm);
      if (warp_id() == 0) {
        const int count = min(keep_count<T>(S.lam, S.perm, n2, kmax, P.cutoff, P.delta), kmax);
        if (tid() == 0) S.misc[M_KEEP] = count;
      }
      __syncthreads();
      keep = S.misc[M_KEEP];
      if (warp_id() == kWarps - 1) {  // the others go on meanwhile
        const double w = discarded_weight(S.lam, S.perm, n2, keep);
        if (lane_id() == 0) S.dmisc[D_DISC] += w;
      }
      // sorted, kept right singular vectors: Vs[:, c] = V[:, perm[c]], c < keep
      // (or the rotated column of X over its norm)
      for (int e = tid(); e < n2 * keep; e += kThreads) {
        int i = e / keep, c = e % keep;
        cplx<T> v = Vc[static_cast<int64_t>(S.perm[c]) * n2 + i];
        if (vec_from_columns) {
          T l = S.lam[S.perm[c]];
          v = l > T(0) ? cscale(v, T(1) / sqrt(l)) : cmake<T>(i == c ? T(1) : T(0), 0);
        }
        X.vs[i * keep + c] = v;
      }
      __syncthreads();
    }
    // and the new right-canonical site k: B[c][s][r] = conj(Vs[(s*kappa + r)][c]).
    // Vectors rounded to float from a higher precision are orthonormal to rounding
    // (from pairs of floats, svd_small has stored the site too); the others take one
    // Newton-Schulz step before.
    if (!rounded) reorthonormalize<T>(n2, keep, X.vs, X.e, X.y, S.tile);
    if (!rounded || !svd64) {
      for (int e = tid(); e < keep * n2; e += kThreads) {
        int c = e / n2, sr = e % n2;
        Bk[e] = cconj(X.vs[sr * keep + c]);
      }
    }
    // W = M Vs (Dl x keep)
    cgemm<T, 0, 0>(Dl, keep, n2, one, M, n2, X.vs, keep, zero, X.w, keep, S.tile);
    // M_{k-1} = A'_{k-1} (left reshape 2D_{k-1} x Dl) W
    const int Dll = Dbond(k - 1);
    const cplx<T> *Akm1 = X.ap + S.off[k - 1 - a];
    cgemm<T, 0, 0>(2 * Dll, keep, Dl, one, Akm1, Dl, X.w, keep, zero, X.mbuf, keep, S.tile);
    if (tid() == 0) {
      chi[k] = keep;
      tally(S.dmisc, D_FLOPS) += gemm_flops(Dl, keep, n2) + gemm_flops(2 * Dll, keep, Dl);
    }
    __syncthreads();
    M = X.mbuf;
    kappa = keep;
  }
  prof_mark(S.dmisc, PROF_RIGHT, tp);
  // centre site a = M (chi[a] x 2 x kappa), renormalised
  cplx<T> *Aa = site_ptr<T>(P, shot, a);
  const int64_t tot = static_cast<int64_t>(chi[a]) * 2 * kappa;
  double nrm = 0;
  for (int64_t e = tid(); e < tot; e += kThreads) nrm += cabs2d(M[e]);
  nrm = block_sum(nrm, S.red);
  T inv = static_cast<T>(nrm > 0 ? 1.0 / sqrt(nrm) : 0.0);
  for (int64_t e = tid(); e < tot; e += kThreads) Aa[e] = cscale(M[e], inv);
  if (tid() == 0) {
    if (!(nrm > 0) || !isfinite(nrm)) S.misc[M_FAIL] = STN_ENUMERIC;
    S.misc[M_CENTER] = a;
    int mx = S.misc[M_MAXCHI];
    for (int k = a + 1; k <= b; ++k) mx = max(mx, chi[k]);
    S.misc[M_MAXCHI] = mx;
  }
  __syncthreads();
}

// <phi| i^m X^x Z^z |phi> over sites [a, b] (centre inside, so the rest of
// the chain contracts to the identity).  Returns the real part.
template <typename T>
static __device__ __noinline__ double mps_expect(const EngineParams &P, const Smem<T> &S, int64_t shot,
                             const Scratch<T> &X, int a, int b, int m) {
  const int *chi = S.chi;
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  MpoSpec<T> sp;
  sp.kind = MPO_ROT; sp.lo = -1; sp.hi = -1; sp.j = -1;
  sp.w0 = one; sp.w1 = one; sp.v0 = zero; sp.v1 = zero;
  for (int k = a; k <= b; ++k) {
    const cplx<T> *A = site_ptr<T>(P, shot, k);
    const int cl = chi[k], cr = chi[k + 1];
    // SA = (X^x Z^z)_k A_k
    cplx<T> op[4];
    site_op(sp, S.ppx, S.ppz, k, 1, op);
    const int64_t tot = static_cast<int64_t>(cl) * 2 * cr;
    for (int64_t e = tid(); e < tot; e += kThreads) {
      int r = static_cast<int>(e % cr), s = static_cast<int>((e / cr) % 2);
      int64_t l = e / (2 * cr);
      cplx<T> v = cmake<T>(0, 0);
      cfma(v, op[s * 2 + 0], A[(l * 2 + 0) * cr + r]);
      cfma(v, op[s * 2 + 1], A[(l * 2 + 1) * cr + r]);
      X.sa[e] = v;
    }
    __syncthreads();
    if (k == a) {
      cgemm<T, 1, 0>(cr, cr, 2 * cl, one, A, cr, X.sa, cr, zero, X.e, cr, S.tile);
      if (tid() == 0) tally(S.dmisc, D_FLOPS) += gemm_flops(cr, cr, 2 * cl);
    } else {
      cgemm<T, 0, 0>(cl, 2 * cr, cl, one, X.e, cl, X.sa, 2 * cr, zero, X.te, 2 * cr, S.tile);
      cgemm<T, 1, 0>(cr, cr, 2 * cl, one, A, cr, X.te, cr, zero, X.e, cr, S.tile);
      if (tid() == 0) tally(S.dmisc, D_FLOPS) += gemm_flops(cl, 2 * cr, cl) + gemm_flops(cr, cr, 2 * cl);
    }
  }
  const int cb = chi[b + 1];
  double re = 0, im = 0;
  for (int i = tid(); i < cb; i += kThreads) {
    re += static_cast<double>(X.e[i * cb + i].re);
    im += static_cast<double>(X.e[i * cb + i].im);
  }
  re = block_sum(re, S.red);
  im = block_sum(im, S.red);
  // multiply by i^m, keep the real part
  switch (m & 3) {
    case 0: return re;
    case 1: return -im;
    case 2: return -re;
    default: return im;
  }
}

// ---------------------------------------------------------------------------
// Tableau helpers (shared memory, one thread unless noted).
static __device__ __forceinline__ int popc64(uint64_t v) { return __popcll(v); }

// row r <- row r * row s (Pauli product with the exact phase)
static __device__ void row_mul(uint64_t *tx, uint64_t *tz, uint8_t *tm, int W, int r, int s) {
  int sw = 0;
  for (int w = 0; w < W; ++w) {
    sw += popc64(tz[r * W + w] & tx[s * W + w]);
    tx[r * W + w] ^= tx[s * W + w];
    tz[r * W + w] ^= tz[s * W + w];
  }
  tm[r] = static_cast<uint8_t>((tm[r] + tm[s] + 2 * sw) & 3);
}

// rows of X errors anticommute with Z_q, and vice versa
static __device__ void pauli_left(uint8_t *tm, int n, int q, int letter /*1 X, 2 Y, 3 Z*/) {
  if (letter == 1 || letter == 2) tm[n + q] = static_cast<uint8_t>((tm[n + q] + 2) & 3);
  if (letter == 3 || letter == 2) tm[q] = static_cast<uint8_t>((tm[q] + 2) & 3);
}

// P' = row r1 * row r2 (r2 < 0: just row r1) into ppx/ppz, phase returned
static __device__ int conj_rows(const uint64_t *tx, const uint64_t *tz, const uint8_t *tm, int W, int r1,
                         int r2, uint64_t *ppx, uint64_t *ppz) {
  int m = tm[r1];
  int sw = 0;
  for (int w = 0; w < W; ++w) {
    ppx[w] = tx[r1 * W + w];
    ppz[w] = tz[r1 * W + w];
    if (r2 >= 0) {
      sw += popc64(ppz[w] & tx[r2 * W + w]);
      ppx[w] ^= tx[r2 * W + w];
      ppz[w] ^= tz[r2 * W + w];
    }
  }
  if (r2 >= 0) m += tm[r2] + 2 * sw;
  return m & 3;
}

// Single-qubit Clifford L applied to the site-j letter of every row:
// R -> L R L^dag, for the four L that take the measured eigenvector to |0>:
// index 0: X,+1 (H)  1: X,-1 (X H)  2: Y,+1 (H S^dag)  3: Y,-1 (X H S^dag).
// Table: [L][xz] -> (x', z', dm) with xz = 2x + z.
__constant__ uint8_t kLTable[4][4][3] = {
    {{0, 0, 0}, {1, 0, 0}, {0, 1, 0}, {1, 1, 2}},
    {{0, 0, 0}, {1, 0, 0}, {0, 1, 2}, {1, 1, 0}},
    {{0, 0, 0}, {1, 0, 0}, {1, 1, 1}, {0, 1, 3}},
    {{0, 0, 0}, {1, 0, 0}, {1, 1, 3}, {0, 1, 1}},
};

// C <- C U L^dag for U = prod_{k != j} controlled-P'_k (control j): every row
// R -> L (U R U) L^dag, with U R U = R Z_j^a (x_j(R) = 0) or
// (-1)^a R Z_j^a Q (x_j(R) = 1), a = [R anticommutes with Q],
// Q = prod_{k != j} P'_k.  CTA-wide over rows.
static __device__ void tableau_caseB(uint64_t *tx, uint64_t *tz, uint8_t *tm, int n, int W,
                              const uint64_t *ppx, const uint64_t *ppz, int j, int lidx) {
  const int jw = j >> 6;
  const uint64_t jb = 1ull << (j & 63);
  for (int r = tid(); r < 2 * n; r += kThreads) {
    int an = 0, mq = 0;
    for (int w = 0; w < W; ++w) {
      uint64_t xq = ppx[w] & (w == jw ? ~jb : ~0ull);
      uint64_t zq = ppz[w] & (w == jw ? ~jb : ~0ull);
      an += popc64((tx[r * W + w] & zq) ^ (tz[r * W + w] & xq));
      mq += popc64(xq & zq);
    }
    an &= 1;
    const bool xj = (tx[r * W + jw] & jb) != 0;
    int m = tm[r];
    if (an) tz[r * W + jw] ^= jb;
    if (xj) {
      if (an) m += 2;
      int sw = 0;
      for (int w = 0; w < W; ++w) {
        uint64_t xq = ppx[w] & (w == jw ? ~jb : ~0ull);
        uint64_t zq = ppz[w] & (w == jw ? ~jb : ~0ull);
        sw += popc64(tz[r * W + w] & xq);
        tx[r * W + w] ^= xq;
        tz[r * W + w] ^= zq;
      }
      m += mq + 2 * sw;
    }
    int x = (tx[r * W + jw] & jb) ? 1 : 0, z = (tz[r * W + jw] & jb) ? 1 : 0;
    const uint8_t *e = kLTable[lidx][2 * x + z];
    if (e[0]) tx[r * W + jw] |= jb; else tx[r * W + jw] &= ~jb;
    if (e[1]) tz[r * W + jw] |= jb; else tz[r * W + jw] &= ~jb;
    tm[r] = static_cast<uint8_t>((m + e[2]) & 3);
  }
  __syncthreads();
}

// Projector MPO of outcome `bit` for the measured P' (thread 0): case A
// (no X or Y in P') projects with (I + (-1)^bit P')/2; case B applies the
// controlled-Pauli product with the site-j projection onto the lambda
// eigenvector, lambda = (-1)^bit * sign(P').
template <typename T>
static __device__ void set_meas_spec(const Smem<T> &S, int bit) {
  MpoSpec<T> &sp = *S.spec;
  const int mb = S.misc[M_BIT];
  const int m = mb & 3;
  const int neg = (mb >> 4) & 1;
  if (!S.misc[M_CASEB]) {
    // P' = i^m Z^z with m even (Hermitian, no X): keep the states whose S
    // parity makes (-1)^b i^m (-1)^parity = +1
    sp.kind = MPO_PROJ_Z;
    const int sgn = (bit ? -1 : 1) * ((m & 2) ? -1 : 1);
    sp.par = sgn > 0 ? 0 : 1;
    sp.w0 = cmake<T>(1, 0);
    sp.w1 = cmake<T>(1, 0);
  } else {
    const int jq = S.misc[M_J];
    const bool zj = (S.ppz[jq >> 6] >> (jq & 63)) & 1;
    int lam = (bit ? -1 : 1) * (neg ? -1 : 1);
    const T r2 = static_cast<T>(0.70710678118654752440);
    sp.kind = MPO_PROJ_B;
    sp.w0 = cmake<T>(1, 0);
    sp.w1 = cmake<T>(1, 0);
    sp.v0 = cmake<T>(r2, 0);
    sp.v1 = zj ? cmake<T>(0, lam > 0 ? r2 : -r2) : cmake<T>(lam > 0 ? r2 : -r2, 0);
    S.misc[M_LIDX] = (zj ? 2 : 0) + (lam < 0 ? 1 : 0);
  }
}

// ---------------------------------------------------------------------------
// B: resident CTAs per SM the registers are allotted for.  With 256 threads and
// one CTA per SM (a batch of up to one shot per SM) the 255 registers a thread
// may then use save spills: 5 % of a d = 5 round against B = 2.
template <typename T, int B>
__global__ void __launch_bounds__(kThreads, B) round_kernel(EngineParams P) {
  extern __shared__ __align__(16) char smem_raw[];
  const int n = P.n, W = P.W;
  Smem<T> S = carve<T>(smem_raw, n, W, P.svd_elems);
  Scratch<T> X = scratch_for<T>(P, P.work_c);
  // complex64 with use_tc (gemm_units = STN_GEMM_TENSOR): the large
  // contractions run on the tensor cores, staged in the shared SVD buffer
  // (free whenever a GEMM runs)
  bool tc_alloc = false;
  if constexpr (sizeof(T) == 4 && !kLight) tc_alloc = P.use_tc && static_cast<int64_t>(P.svd_elems) * 2 >= kTcStageFloats;
  if (tc_alloc) tc_setup(reinterpret_cast<float *>(S.jbuf));
  else tc_disable();
  bool tc_live = tc_alloc;  // CTA-uniform
  // With a ticket counter the CTAs take the batch's shots in order as they
  // finish (a work queue that balances uneven shots when the batch holds
  // more shots than CTAs); without one, shots are grid-strided.
  for (int64_t it = 0;; ++it) {
    int64_t shot = blockIdx.x + it * gridDim.x;
    if (P.ticket) {
      if (tid() == 0) S.misc[M_TICKET] = atomicAdd(P.ticket, 1);
      __syncthreads();
      shot = S.misc[M_TICKET];
      __syncthreads();
    }
    if (shot >= P.shots) break;
    // load the frame and the MPS bookkeeping
    for (int e = tid(); e < 2 * n * W; e += kThreads) {
      S.tx[e] = P.tab_x[shot * 2 * n * W + e];
      S.tz[e] = P.tab_z[shot * 2 * n * W + e];
    }
    for (int e = tid(); e < 2 * n; e += kThreads) S.tm[e] = P.tab_m[shot * 2 * n + e];
    for (int e = tid(); e <= n; e += kThreads) S.chi[e] = P.chi[shot * (n + 1) + e];
    if (tid() == 0) {
      S.misc[M_CENTER] = P.center[shot];
      S.misc[M_FAIL] = P.status[shot];
      S.misc[M_MAXCHI] = P.maxchi[shot];
      S.dmisc[D_DISC] = P.disc[shot];
      S.dmisc[D_LOGP] = P.logp[shot];
      tally(S.dmisc, D_FLOPS) = 0;
      for (int i = 0; i < kProfSlots; ++i) tally(S.dmisc, D_PROF + 1 + i) = 0;
    }
    __syncthreads();
    long long t_ops = clock64();
    const uint64_t gshot = (P.shot_offset_dev ? *P.shot_offset_dev : P.shot_offset) + static_cast<uint64_t>(shot);
    for (int oi = P.op_begin; oi < P.op_end; ++oi) {
      if (tc_live) {
        // a tensor-core wait ran out: this shot stops, the rest use the CUDA
        // cores.  Every thread reads the flag before thread 0 may clear it.
        const int tc_failed = g_tc.failed;
        __syncthreads();
        if (tc_failed) {
          if (tid() == 0) {
            S.misc[M_FAIL] = STN_ETIMEOUT;
            g_tc.failed = 0;
            g_tc.enabled = 0;
          }
          tc_live = false;
          __syncthreads();
        }
      }
      if (S.misc[M_FAIL]) break;
      const Op op = P.ops[oi];
      switch (op.kind) {
        case OP_RESET_FLIP:
          if (tid() == 0 && philox_uniform(P.seed, gshot, op.ev) < P.pR) pauli_left(S.tm, n, op.a, 1);
          break;
        case OP_H:
          if (tid() < W) {
            int w = tid();
            uint64_t t = S.tx[op.a * W + w];
            S.tx[op.a * W + w] = S.tx[(n + op.a) * W + w];
            S.tx[(n + op.a) * W + w] = t;
            t = S.tz[op.a * W + w];
            S.tz[op.a * W + w] = S.tz[(n + op.a) * W + w];
            S.tz[(n + op.a) * W + w] = t;
          }
          if (tid() == 0) {
            uint8_t t = S.tm[op.a];
            S.tm[op.a] = S.tm[n + op.a];
            S.tm[n + op.a] = t;
          }
          break;
        case OP_NOISE1:
          if (tid() == 0) {
            double u = philox_uniform(P.seed, gshot, op.ev);
            if (u < P.p1) pauli_left(S.tm, n, op.a, 1 + min(2, static_cast<int>(3.0 * u / P.p1)));
          }
          break;
        case OP_CNOT:
          if (tid() == 0) {
            row_mul(S.tx, S.tz, S.tm, W, op.a, op.b);          // X_c <- X_c X_t
            row_mul(S.tx, S.tz, S.tm, W, n + op.b, n + op.a);  // Z_t <- Z_t Z_c (rows commute)
          }
          break;
        case OP_NOISE2:
          if (tid() == 0) {
            double u = philox_uniform(P.seed, gshot, op.ev);
            if (u < P.p2) {
              int idx = min(14, static_cast<int>(15.0 * u / P.p2)) + 1;
              int lc = idx / 4, lt = idx % 4;  // 0 I, 1 X, 2 Y, 3 Z
              if (lc) pauli_left(S.tm, n, op.a, lc);
              if (lt) pauli_left(S.tm, n, op.b, lt);
            }
          }
          break;
        case OP_ROT:
        case OP_MEAS: {
          const bool meas = op.kind == OP_MEAS;
          if (tid() == 0) {
            int m;
            if (meas) m = conj_rows(S.tx, S.tz, S.tm, W, n + op.a, -1, S.ppx, S.ppz);
            else if (op.pauli == 0) m = conj_rows(S.tx, S.tz, S.tm, W, n + op.a, n + op.b, S.ppx, S.ppz);
            else m = conj_rows(S.tx, S.tz, S.tm, W, op.a, op.b, S.ppx, S.ppz);
            int lo = n, hi = -1, j = -1, xz = 0;
            for (int w = 0; w < W; ++w) {
              const uint64_t x = S.ppx[w], any = x | S.ppz[w];
              if (any) {
                if (hi < 0) lo = 64 * w + __ffsll(any) - 1;
                hi = 64 * w + 63 - __clzll(any);
              }
              if (x && j < 0) j = 64 * w + __ffsll(x) - 1;
              xz += popc64(x & S.ppz[w]);
            }
            const int xany = j >= 0;
            S.misc[M_LO] = lo;
            S.misc[M_HI] = hi;
            S.misc[M_A] = lo;
            S.misc[M_B] = hi;
            S.misc[M_J] = j;
            S.misc[M_CASEB] = xany;
            S.misc[M_BIT] = m | ((((m - xz) & 3) == 2) << 4);  // phase | (sign < 0) << 4
            MpoSpec<T> &sp = *S.spec;
            sp.lo = lo; sp.hi = hi; sp.j = j;
            if (!meas) {
              double sn, cs;
              sincos(P.theta[op.idx], &sn, &cs);
              cplx<T> w1 = cmul(cmake<T>(0, static_cast<T>(-sn)), ipow<T>(m));
              sp.kind = MPO_ROT;
              sp.w0 = cmake<T>(static_cast<T>(cs), 0);
              sp.w1 = w1;
            }
            if (lo > hi) S.misc[M_FAIL] = STN_ENUMERIC;  // identity Pauli cannot occur
            if (P.tape_info) {
              const int64_t t = shot * P.n_ops_total + oi;
              for (int w = 0; w < W; ++w) {
                P.tape_px[t * W + w] = S.ppx[w];
                P.tape_pz[t * W + w] = S.ppz[w];
              }
              int32_t *ti = P.tape_info + t * kTapeInts;
              ti[0] = m & 3;
              ti[1] = lo;
              ti[2] = hi;
              ti[3] = j;
            }
          }
          __syncthreads();
          if (S.misc[M_FAIL]) break;
          const int a = S.misc[M_A], b = S.misc[M_B];
          {
            // the centre moves into [a, b] by exact gauge steps; the sweep
            // then covers the operator's support only
            const int c0 = S.misc[M_CENTER];
            const int tgt = c0 < a ? a : (c0 > b ? b : c0);
            if (tgt != c0) {
              long long tg = clock64();
              mps_move_center<T>(P, S, shot, X, tgt);
              prof_mark(S.dmisc, PROF_GAUGE, tg);
            }
          }
          if (S.misc[M_FAIL]) break;
          int caseB = 0, lidx = 0, outcome = 0;
          if (meas) {
            // The Born probability of the less likely branch is the squared
            // norm of its projected state, from R factors: any deviation of
            // the sites outside [a, b] from exact isometries (rounding of the
            // gauge steps and sweeps) changes it only relatively.  The
            // expectation value only decides which branch that is.
            const int mb = S.misc[M_BIT];
            long long tq = clock64();
            const double e = mps_expect<T>(P, S, shot, X, a, b, mb & 3);
            const int small = e >= 0.0 ? 1 : 0;
            if (tid() == 0) set_meas_spec<T>(S, small);
            __syncthreads();
            prof_mark(S.dmisc, PROF_EXPECT, tq);
            const double ps = fmin(1.0, fmax(0.0, mps_prepare<T>(P, S, shot, X, a, b, true)));
            prof_mark(S.dmisc, PROF_LEFT, tq);
            if (tid() == 0) {
              double p0 = small == 0 ? ps : 1.0 - ps;
              double u = philox_uniform(P.seed, gshot, op.ev);
              const int flip = philox_uniform(P.seed, gshot, op.ev + 1) < P.pM ? 1 : 0;
              int bit = u < p0 ? 0 : 1;
              if (P.forced)  // adjoint forward pass: the outcome that reproduces the record
                bit = ((P.forced[shot * P.rec_bytes + op.idx / 8] >> (op.idx % 8)) & 1) ^ flip;
              double pb = bit == 0 ? p0 : 1.0 - p0;
              if (!P.forced && fabs(u - p0) < kNearThreshold) P.near[shot] += 1;
              P.born[shot * P.n_meas + op.idx] = pb;
              S.dmisc[D_LOGP] += log(pb);
              if (bit ^ flip) P.records[shot * P.rec_bytes + op.idx / 8] |= static_cast<uint8_t>(1u << (op.idx % 8));
              S.misc[M_OUTCOME] = bit;
              if (bit != small) set_meas_spec<T>(S, bit);
              if (P.tape_info) {
                int32_t *ti = P.tape_info + (shot * P.n_ops_total + oi) * kTapeInts;
                const int mb = S.misc[M_BIT];
                ti[0] = (mb & 3) | (S.misc[M_CASEB] << 2) | (bit << 3) | (S.misc[M_LIDX] << 4) |
                        (((mb >> 4) & 1) << 6);
              }
            }
            __syncthreads();
            caseB = S.misc[M_CASEB];
            lidx = S.misc[M_LIDX];
            outcome = S.misc[M_OUTCOME];
            tq = clock64();
            if (outcome != small) mps_prepare<T>(P, S, shot, X, a, b, false);
            __syncthreads();
            prof_mark(S.dmisc, PROF_LEFT, tq);
            mps_finish<T>(P, S, shot, X, a, b);
          } else {
            long long tq = clock64();
            mps_prepare<T>(P, S, shot, X, a, b, false);
            __syncthreads();
            prof_mark(S.dmisc, PROF_LEFT, tq);
            mps_finish<T>(P, S, shot, X, a, b);
            if (P.phi_store && P.rot_ord[oi] >= 0) {  // adjoint: keep the state after the rotation
              const int64_t slot = shot * P.n_rot + P.rot_ord[oi];
              cplx<T> *dst = reinterpret_cast<cplx<T> *>(P.phi_store) + slot * P.slab_elems;
              for (int k = 0; k < n; ++k) {
                const cplx<T> *src = site_ptr<T>(P, shot, k);
                const int64_t cnt = 2ll * S.chi[k] * S.chi[k + 1];
                for (int64_t e = tid(); e < cnt; e += kThreads) dst[P.site_off[k] + e] = src[e];
              }
              for (int e = tid(); e <= n; e += kThreads) P.phi_chi[slot * (n + 1) + e] = S.chi[e];
            }
          }
          if (meas) {
            if (caseB) tableau_caseB(S.tx, S.tz, S.tm, n, W, S.ppx, S.ppz, S.misc[M_J], lidx);
            if (tid() == 0 && op.pauli == 1) {
              if (outcome) pauli_left(S.tm, n, op.a, 1);
              if (philox_uniform(P.seed, gshot, op.ev + 2) < P.pR) pauli_left(S.tm, n, op.a, 1);
            }
          }
          break;
        }
        default:
          if (tid() == 0) S.misc[M_FAIL] = STN_EINVAL;
      }
      __syncthreads();
    }
    // store
    for (int e = tid(); e < 2 * n * W; e += kThreads) {
      P.tab_x[shot * 2 * n * W + e] = S.tx[e];
      P.tab_z[shot * 2 * n * W + e] = S.tz[e];
    }
    for (int e = tid(); e < 2 * n; e += kThreads) P.tab_m[shot * 2 * n + e] = S.tm[e];
    for (int e = tid(); e <= n; e += kThreads) P.chi[shot * (n + 1) + e] = S.chi[e];
    if (tid() == 0) {
      P.center[shot] = S.misc[M_CENTER];
      P.status[shot] = S.misc[M_FAIL];
      P.maxchi[shot] = S.misc[M_MAXCHI];
      P.disc[shot] = S.dmisc[D_DISC];
      P.logp[shot] = S.dmisc[D_LOGP];
      P.flops[shot] += static_cast<double>(tally(S.dmisc, D_FLOPS)) / 3.0;
      tally(S.dmisc, D_PROF + 1 + PROF_OPS) = clock64() - t_ops;
      for (int i = 0; i < kProfSlots; ++i)
        P.prof[shot * kProfSlots + i] += static_cast<double>(tally(S.dmisc, D_PROF + 1 + i));
      if (S.misc[M_FAIL]) atomicCAS(P.err, 0, S.misc[M_FAIL]);
    }
    __syncthreads();
  }
  if (tc_alloc) tc_teardown();
}

// Identity frame, |0...0>, cleared records and accumulators.
template <typename T>
__global__ void init_kernel(EngineParams P) {
  const int n = P.n, W = P.W;
  for (int64_t shot = blockIdx.x; shot < P.shots; shot += gridDim.x) {
    for (int e = tid(); e < 2 * n * W; e += blockDim.x) {
      int r = e / W, w = e % W;
      int q = r % n;
      uint64_t bit = (q >> 6) == w ? (1ull << (q & 63)) : 0ull;
      P.tab_x[shot * 2 * n * W + e] = r < n ? bit : 0ull;
      P.tab_z[shot * 2 * n * W + e] = r < n ? 0ull : bit;
    }
    for (int e = tid(); e < 2 * n; e += blockDim.x) P.tab_m[shot * 2 * n + e] = 0;
    for (int e = tid(); e <= n; e += blockDim.x) P.chi[shot * (n + 1) + e] = 1;
    cplx<T> *slab = reinterpret_cast<cplx<T> *>(P.mps) + shot * P.slab_elems;
    for (int k = tid(); k < n; k += blockDim.x) {
      slab[P.site_off[k]] = cmake<T>(1, 0);
      slab[P.site_off[k] + 1] = cmake<T>(0, 0);
    }
    for (int e = tid(); e < P.rec_bytes; e += blockDim.x) P.records[shot * P.rec_bytes + e] = 0;
    for (int e = tid(); e < P.n_meas; e += blockDim.x) P.born[shot * P.n_meas + e] = 0.0;
    if (tid() == 0) {
      P.center[shot] = 0;
      P.status[shot] = 0;
      P.maxchi[shot] = 1;
      P.near[shot] = 0;
      P.disc[shot] = 0.0;
      P.logp[shot] = 0.0;
    }
  }
}

// ---------------------------------------------------------------------------
// The truncation sweep's SVD on its own: right singular vectors V (n x n,
// column-major; columns from min(m, n) on, or beyond the rank, are zero) and
// squared singular values of the row-major m x n matrix A.  complex128 whose
// matrix fits shared memory: svd_small on A.  Else, on the copy in `work`
// (work may be A): R factor, Jacobi on X = R^dag (n x k), V = normalised
// columns of X; with CL by the CTAs of a cluster.
template <typename T>
__host__ __device__ __forceinline__ bool svd_bond_small(int m, int n) {
  return sizeof(T) == 8 && n <= kSmallSvdCols && n * (m | 1) <= SvdSmem<T>::elems;
}

template <typename T, bool CL>
static __device__ void svd_bond(int m, int n, const cplx<T> *A, cplx<T> *work, cplx<T> *V, T *sig2, cplx<T> *buf,
                                cplx<T> *uv, double *red, int *flag, float *rv_wrk) {
  if constexpr (sizeof(T) == 8 && !CL) {
    if (svd_bond_small<T>(m, n)) {
      const int rank = svd_small<T, true>(m, n, A, V, sig2, 0.0, buf, uv, red);
      for (int e = tid() + rank * n; e < n * n; e += kThreads) V[e] = cmake<T>(0, 0);
      return;
    }
  }
  const int t0 = tid() + kThreads * share_rank<CL>(), step = kThreads * share_size<CL>();
  // complex128 matrices that svd_small would take whatever their scale: to entries
  // around 1, by a power of two that every CTA finds for itself
  T down = 1, up = 1;
  if constexpr (sizeof(T) == 8 && CL) {
    int *top = reinterpret_cast<int *>(red);
    if (tid() == 0) *top = 0;
    __syncthreads();
    int hi = 0;
    for (int e = tid(); e < m * n; e += kThreads)
      hi = max(hi, max(__double2hiint(A[e].re) & 0x7fffffff, __double2hiint(A[e].im) & 0x7fffffff));
    hi = __reduce_max_sync(0xffffffffu, hi);
    if (lane_id() == 0) atomicMax(top, hi);
    __syncthreads();
    const int ex = min(2045, max(1, *top >> 20));
    down = __hiloint2double((2046 - ex) << 20, 0);
    up = __hiloint2double(ex << 20, 0);
    share_sync<CL>();  // A may be work
  }
  if (work != A || CL)
    for (int e = t0; e < m * n; e += step) work[e] = cscale(A[e], down);
  share_sync<CL>();
  qr_r_inplace<T, CL>(m, n, work, n, buf, SvdSmem<T>::elems);
  const int k = min(m, n);
  const bool regs = sizeof(T) == 4 && k > 16 && n <= kThreads;
  const bool x_smem = !CL && !regs && n * k <= SvdSmem<T>::elems;
  cplx<T> *Xc = x_smem ? buf : work;
  for (int e = t0; e < n * k; e += step) Xc[e] = cconj(work[e]);
  share_sync<CL>();
  if (x_smem) svd_onesided<T>(n, k, Xc, nullptr, sig2, flag, red);
  else svd_onesided_blocked<T, CL>(n, k, Xc, nullptr, sig2, flag, red, buf, SvdSmem<T>::elems, regs ? rv_wrk : nullptr);
  for (int e = t0; e < n * n; e += step) {
    const int c = e / n;
    const T l = c < k ? sig2[c] : T(0);
    V[e] = l > T(0) ? cscale(Xc[e], T(1) / sqrt(l)) : cmake<T>(0, 0);
  }
  if (CL) share_sync<CL>();
  if constexpr (sizeof(T) == 8 && CL)
    for (int c = t0; c < k; c += step) sig2[c] = sig2[c] * up * up;
  for (int c = k + t0; c < n; c += step) sig2[c] = T(0);
  if (CL) share_sync<CL>();  // no CTA leaves while another may read its shared memory
}

// R factor or SVD of one large matrix that is called alone, by a cluster of CTAs.
// One CTA left the GPU idle: its block pairs take turns although a round's are
// disjoint.  Eight CTAs (the portable limit) have a block pair of 16 + 16 columns
// each up to 256 columns, and in complex128 blocks of a sixteenth of the columns.
// The same code on one CTA and on eight: a 256 x 192 complex64 SVD 21.8 and 4.57 ms,
// 60 x 50 2.07 and 1.16 ms; complex128 128 x 128 58 and 10.6 ms, 72 x 66 (svd_small on
// one CTA, bound by its SM's FP64 rate) 7.3 and 4.3 ms; the R factor of 512 x 250 in
// complex64 2.76 and 1.37 ms, of 200 x 100 in complex128 3.8 and 1.8 ms.
// From 48 columns on: 64 x 48 takes 2.65 and 2.33 ms in complex128 and 1.26 and 1.05 ms
// in complex64; 52 x 40 1.66 and 1.83 ms in complex128 (1.10 and 0.97 ms in complex64,
// which could start lower: 40 x 32 0.57 and 0.49 ms).
constexpr int kShareCtas = 8;
constexpr int kShareMinCols = 48;

struct DenseSmem {
  double *red;
  int *flag;
  char *uv, *buf;
  float *rv_wrk;
};
template <typename T>
static __device__ DenseSmem dense_smem(char *base) {
  DenseSmem s;
  s.red = reinterpret_cast<double *>(base);
  s.flag = reinterpret_cast<int *>(s.red + kRedDoubles + 16);
  s.uv = reinterpret_cast<char *>(s.flag + 16);
  s.buf = s.uv + sizeof(cplx<T>) * kMaxVec;
  s.rv_wrk = reinterpret_cast<float *>(s.buf + sizeof(cplx<T>) * SvdSmem<T>::elems);
  return s;
}
template <typename T>
static size_t dense_smem_bytes() {
  size_t smem = sizeof(double) * (kRedDoubles + 16) + sizeof(int) * 16 + sizeof(cplx<T>) * kMaxVec;
  smem += sizeof(cplx<T>) * SvdSmem<T>::elems;  // QR panel, SVD matrix or staged column blocks
  return smem + sizeof(float) * kRvWrkFloats;   // register-visit reductions
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) dense_shared_kernel(bool svd, int m, int n, cplx<T> *A, cplx<T> *work,
                                                                   cplx<T> *V, T *sig2) {
  extern __shared__ __align__(16) char smem_raw[];
  tc_disable();
  const DenseSmem s = dense_smem<T>(smem_raw);
  cplx<T> *buf = reinterpret_cast<cplx<T> *>(s.buf);
  if (svd) svd_bond<T, true>(m, n, A, work, V, sig2, buf, reinterpret_cast<cplx<T> *>(s.uv), s.red, s.flag, s.rv_wrk);
  else qr_r_inplace<T, true>(m, n, A, n, buf, SvdSmem<T>::elems);
}

template <typename T>
static cudaError_t launch_dense_shared(bool svd, int m, int n, cplx<T> *A, cplx<T> *work, cplx<T> *V, T *sig2,
                                       cudaStream_t s) {
  const size_t smem = dense_smem_bytes<T>();
  cudaError_t e = cudaFuncSetAttribute(dense_shared_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(kShareCtas);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = kShareCtas;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, dense_shared_kernel<T>, svd, m, n, A, work, V, sig2);
}

// Which R factors called alone take qr_small: none in complex64, where the phase of
// a row is known to 1e-3 at worst and moves with every order of summation: their R
// is qr_r_inplace's whatever the size, and its unit reflectors take columns of 1e8
// beside ones of 1e33.  (A 40 x 20 one: 47 us against 29 by qr_small, 159 by the
// panels of one column after the other.)
template <typename T>
__host__ __device__ __forceinline__ bool qr_alone_small(int m, int n, bool with_q) {
  return sizeof(T) == 8 && qr_small_elems(m, n, with_q) <= SvdSmem<T>::elems;
}

// Whether qr_small takes the entries of a caller's complex128 matrix.  CTA-wide.
template <typename T>
static __device__ __forceinline__ bool in_small_range(int count, const cplx<T> *A) {
  bool large = false;
  if constexpr (sizeof(T) == 8)
    for (int e = tid(); e < count; e += kThreads)
      large |= max(__double2hiint(A[e].re) & 0x7fffffff, __double2hiint(A[e].im) & 0x7fffffff) >= (1023 + 300) << 20;
  return !__syncthreads_or(large);
}

// Which calls a cluster takes.
template <typename T>
static bool shares_svd(int m, int n) {
  return (m < n ? m : n) >= kShareMinCols;
}
template <typename T>
static bool shares_qr(int m, int n) {
  return !qr_alone_small<T>(m, n, false) && (m < n ? m : n) >= kShareMinCols;
}

// Kernel-level checks of the dense routines on one CTA (complex elements of
// precision T, column-major C/V for the SVD, row-major B for the QR).
template <typename T>
__global__ void __launch_bounds__(kThreads, 1) dense_check_kernel(int what, int m, int n, cplx<T> *A,
                                                                  cplx<T> *V, T *sig2, int use_smem) {
  extern __shared__ __align__(16) char smem_raw[];
  tc_disable();
  const DenseSmem s = dense_smem<T>(smem_raw);
  cplx<T> *buf = reinterpret_cast<cplx<T> *>(s.buf);
  double *red = s.red;
  int *flag = s.flag;
  if (what == 0) {
    if (qr_alone_small<T>(m, n, false) && in_small_range(m * n, A)) qr_small<T>(m, n, A, n, false, A, m, nullptr, buf);
    else qr_r_inplace<T>(m, n, A, n, buf, SvdSmem<T>::elems);
  } else if (what == 2) {
    // explicit Q of the gauge steps: reflectors kept in sig2's buffer
    cplx<T> *vstore = reinterpret_cast<cplx<T> *>(sig2);
    if (qr_alone_small<T>(m, n, true) && in_small_range(m * n, A)) {
      qr_small<T>(m, n, A, n, false, A, m, V, buf);
      const int ld = m | 1, steps = min(m, n);
      const ColumnHead<T> *head = reinterpret_cast<const ColumnHead<T> *>(buf + n * ld);
      for (int e = tid(); e < m * steps; e += kThreads) {  // unit vectors there, v with beta here
        const int i = e / steps, c = e % steps;
        if (i >= c) vstore[e] = cscale(i == c ? head[c].v0 : buf[c * ld + i], sqrt(head[c].beta * T(0.5)));
      }
    } else {
      qr_r_inplace<T>(m, n, A, n, buf, SvdSmem<T>::elems, vstore);
      form_q<T>(m, min(m, n), vstore, V, buf, SvdSmem<T>::elems);
    }
  } else if (use_smem == 3) {
    svd_bond<T, false>(m, n, A, A, V, sig2, buf, reinterpret_cast<cplx<T> *>(s.uv), red, flag, s.rv_wrk);
  } else {
    cplx<T> *C = A, *VV = V;
    if (use_smem == 1) {
      C = buf;
      VV = buf + m * n;
      for (int e = tid(); e < m * n; e += kThreads) C[e] = A[e];
      __syncthreads();
    }
    if (use_smem == 2) svd_onesided_blocked<T>(m, n, C, VV, sig2, flag, red, buf, SvdSmem<T>::elems);
    else svd_onesided<T>(m, n, C, VV, sig2, flag, red);
    if (use_smem == 1) {
      for (int e = tid(); e < m * n; e += kThreads) A[e] = C[e];
      for (int e = tid(); e < n * n; e += kThreads) V[e] = VV[e];
    }
  }
}

template <typename T>
cudaError_t launch_dense_check_t(int what, int m, int n, void *A, void *V, void *sig2, int use_smem,
                                        cudaStream_t s) {
  const bool svd = what == 1 && use_smem == 3;
  if (svd ? shares_svd<T>(m, n) : what == 0 && shares_qr<T>(m, n))
    return launch_dense_shared<T>(svd, m, n, static_cast<cplx<T> *>(A), static_cast<cplx<T> *>(A),
                                  static_cast<cplx<T> *>(V), static_cast<T *>(sig2), s);
  const size_t smem = dense_smem_bytes<T>();
  cudaError_t e = cudaFuncSetAttribute(dense_check_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  dense_check_kernel<T><<<1, kThreads, smem, s>>>(what, m, n, static_cast<cplx<T> *>(A),
                                                  static_cast<cplx<T> *>(V), static_cast<T *>(sig2), use_smem);
  return cudaGetLastError();
}

// The sweeps' complex contraction alone: C = alpha op(A) op(B) + beta C through
// cgemm, by one CTA with the tensor cores set up as the round kernel sets them up
// (complex64 and use_tc), else by a CTA per block x block outputs: one CTA for all
// of a 200^3 product took 8.3 ms in complex128 and 351 us in complex64.  *status becomes
// STN_ETIMEOUT if a tensor-core wait ran out.
template <typename T>
__global__ void __launch_bounds__(kThreads, 1) dense_gemm_kernel(int ta, int tb, int m, int n, int k, cplx<T> alpha,
                                                                 const cplx<T> *A, int lda, const cplx<T> *B, int ldb,
                                                                 cplx<T> beta, cplx<T> *C, int ldc, int use_tc,
                                                                 int *status, int block) {
  extern __shared__ __align__(16) char smem_raw[];
  cplx<T> *tile = reinterpret_cast<cplx<T> *>(smem_raw);
  float *stage = reinterpret_cast<float *>(tile + kTileElems);
  bool tc = false;
  if constexpr (sizeof(T) == 4) tc = use_tc != 0;
  if (tc) tc_setup(stage);
  else tc_disable();
  // this CTA's block of C (all of it with the tensor cores)
  const int i0 = blockIdx.x * block, j0 = blockIdx.y * block;
  m = min(block, m - i0);
  n = min(block, n - j0);
  A += ta == 0 ? static_cast<int64_t>(i0) * lda : i0;
  B += tb == 0 ? j0 : static_cast<int64_t>(j0) * ldb;
  C += static_cast<int64_t>(i0) * ldc + j0;
  if (ta == 0 && tb == 0) cgemm<T, 0, 0>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, tile);
  else if (ta == 0) cgemm<T, 0, 1>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, tile);
  else if (tb == 0) cgemm<T, 1, 0>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, tile);
  else cgemm<T, 1, 1>(m, n, k, alpha, A, lda, B, ldb, beta, C, ldc, tile);
  if (tc) {
    if (threadIdx.x == 0 && g_tc.failed) *status = STN_ETIMEOUT;
    tc_teardown();
  }
}

template <typename T>
cudaError_t launch_dense_gemm_t(int ta, int tb, int m, int n, int k, const double *alpha, const void *A, int lda,
                                const void *B, int ldb, const double *beta, void *C, int ldc, int use_tc, int *status,
                                cudaStream_t s) {
  size_t smem = sizeof(cplx<T>) * kTileElems;
  if (sizeof(T) == 4 && use_tc) smem += sizeof(float) * kTcStageFloats;
  cudaError_t e = cudaFuncSetAttribute(dense_gemm_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  cplx<T> al, be;
  al.re = static_cast<T>(alpha[0]);
  al.im = static_cast<T>(alpha[1]);
  be.re = static_cast<T>(beta[0]);
  be.im = static_cast<T>(beta[1]);
  // blocks of 32 x 32 outputs, of 16 x 16 where those would leave SMs without one
  const bool tc = sizeof(T) == 4 && use_tc;
  auto tiles = [&](int b) { return dim3((m + b - 1) / b, (n + b - 1) / b); };
  int block = tc ? (m > n ? m : n) : 32;
  constexpr unsigned kSms = 152;
  if (!tc && tiles(32).x * tiles(32).y < kSms) block = 16;
  dense_gemm_kernel<T><<<tiles(block), kThreads, smem, s>>>(ta, tb, m, n, k, al, static_cast<const cplx<T> *>(A), lda,
                                                 static_cast<const cplx<T> *>(B), ldb, be, static_cast<cplx<T> *>(C),
                                                 ldc, use_tc, status, block);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_init_t(const EngineParams &p, cudaStream_t s) {
  int grid = p.shots < 4096 ? p.shots : 4096;
  if (grid < 1) return cudaSuccess;
  init_kernel<T><<<grid, 128, 0, s>>>(p);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Diagnostics of the current batch, one CTA per shot slot (grid-strided).
// what = DIAG_LOGICAL: out[shot] = <psi| L |psi> for L the product of
//   `letter` (1 X, 3 Z) over the nl qubits lq (Sec. II, Eq. 1: the logical
//   operator's expectation behind the P_L estimator).  L is pushed through
//   the shot's frame, P' = C^dag L C = i^m X^x Z^z (the images of the
//   commuting factors multiplied with the exact phase), the orthogonality
//   centre is moved into P''s support, and <MPS| P' |MPS> is contracted over
//   it.  A shot whose status is set gets NaN.
// what = DIAG_SCHMIDT: for shot `target` only, the centre is moved to site
//   `cut` and the squared singular values of that site as a
//   (2 chi_cut) x chi_{cut+1} matrix, the squared Schmidt coefficients across
//   the cut after site `cut` (Sec. IV B, Fig. 2), go to out[] largest first,
//   their number to *count.
// Both only move the orthogonality centre by exact gauge steps: the state,
// and every later result of the batch, are unchanged (up to rounding).
enum { DIAG_LOGICAL = 0, DIAG_SCHMIDT = 1 };

template <typename T>
__global__ void __launch_bounds__(kThreads, 1) diag_kernel(EngineParams P, int what, int target, int cut,
                                                           const int32_t *lq, int nl, int letter, double *out,
                                                           int *count) {
  extern __shared__ __align__(16) char smem_raw[];
  tc_disable();
  const int n = P.n, W = P.W;
  Smem<T> S = carve<T>(smem_raw, n, W, P.svd_elems);
  Scratch<T> X = scratch_for<T>(P, P.work_c);
  for (int64_t shot = blockIdx.x; shot < P.shots; shot += gridDim.x) {
    if (what == DIAG_SCHMIDT && shot != target) continue;
    for (int e = tid(); e < 2 * n * W; e += kThreads) {
      S.tx[e] = P.tab_x[shot * 2 * n * W + e];
      S.tz[e] = P.tab_z[shot * 2 * n * W + e];
    }
    for (int e = tid(); e < 2 * n; e += kThreads) S.tm[e] = P.tab_m[shot * 2 * n + e];
    for (int e = tid(); e <= n; e += kThreads) S.chi[e] = P.chi[shot * (n + 1) + e];
    if (tid() == 0) {
      S.misc[M_CENTER] = P.center[shot];
      S.misc[M_FAIL] = P.status[shot];
    }
    __syncthreads();
    if (S.misc[M_FAIL]) {
      if (tid() == 0) {
        if (what == DIAG_LOGICAL) out[shot] = nan("");
        else *count = 0;
      }
      __syncthreads();
      continue;
    }
    if (what == DIAG_LOGICAL) {
      if (tid() == 0) {
        for (int w = 0; w < W; ++w) S.ppx[w] = S.ppz[w] = 0;
        int m = 0;
        for (int i = 0; i < nl; ++i) {
          const int r = letter == 3 ? n + lq[i] : lq[i];
          int sw = 0;
          for (int w = 0; w < W; ++w) {
            sw += popc64(S.ppz[w] & S.tx[r * W + w]);
            S.ppx[w] ^= S.tx[r * W + w];
            S.ppz[w] ^= S.tz[r * W + w];
          }
          m += S.tm[r] + 2 * sw;
        }
        int lo = n, hi = -1;
        for (int q = 0; q < n; ++q)
          if (((S.ppx[q >> 6] | S.ppz[q >> 6]) >> (q & 63)) & 1) { lo = min(lo, q); hi = max(hi, q); }
        S.misc[M_LO] = lo;
        S.misc[M_HI] = hi;
        S.misc[M_BIT] = m & 3;
      }
      __syncthreads();
      const int lo = S.misc[M_LO], hi = S.misc[M_HI], m = S.misc[M_BIT];
      double e;
      if (lo > hi) {  // L maps to a multiple of the identity
        e = m == 0 ? 1.0 : (m == 2 ? -1.0 : 0.0);
      } else {
        const int c0 = S.misc[M_CENTER];
        const int tgt = c0 < lo ? lo : (c0 > hi ? hi : c0);
        if (tgt != c0) mps_move_center<T>(P, S, shot, X, tgt);
        e = S.misc[M_FAIL] ? nan("") : mps_expect<T>(P, S, shot, X, lo, hi, m);
      }
      if (tid() == 0) out[shot] = e;
    } else {
      mps_move_center<T>(P, S, shot, X, cut);
      const int l = S.chi[cut], r = S.chi[cut + 1], mrows = 2 * l, kx = min(mrows, r);
      int cnt = 0;
      if (!S.misc[M_FAIL] && mrows <= kMaxVec) {
        const cplx<T> *A = site_ptr<T>(P, shot, cut);
        for (int e = tid(); e < mrows * r; e += kThreads) X.y[e] = A[e];
        __syncthreads();
        qr_r_inplace<T>(mrows, r, X.y, r, S.jbuf, P.svd_elems);
        // Jacobi on R^dag (r x kx, column-major, ld r), in place as in the sweep
        for (int e = tid(); e < r * kx; e += kThreads) X.y[e] = cconj(X.y[e]);
        __syncthreads();
        svd_onesided_blocked<T>(r, kx, X.y, nullptr, X.lam, &S.misc[M_JFLAG], S.red, S.jbuf, P.svd_elems,
                                sizeof(T) == 4 && kx > 16 && r <= kThreads ? reinterpret_cast<float *>(S.lam)
                                                                            : nullptr);
        sort_desc<T>(kx, X.lam, S.perm);
        for (int i = tid(); i < kx; i += kThreads) out[i] = fmax(static_cast<double>(X.lam[S.perm[i]]), 0.0);
        cnt = kx;
      }
      if (tid() == 0) *count = cnt;
    }
    __syncthreads();
    for (int e = tid(); e <= n; e += kThreads) P.chi[shot * (n + 1) + e] = S.chi[e];
    if (tid() == 0) {
      P.center[shot] = S.misc[M_CENTER];
      if (S.misc[M_FAIL]) P.status[shot] = S.misc[M_FAIL];
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// <mu| phase (x)_k op_k |phi> of two MPSs over all n sites: mu is the shot's
// own MPS (bonds S.chi), phi a stored state (sites at site_off in phi, bonds
// phi_chi).  The Pauli string in S.ppx/ppz (letters X^x Z^z) acts on phi when
// with_op.  Transfer matrices E (chi_mu x chi_phi): E <- A_mu^dag (E B),
// through two GEMMs per site.  CTA-wide; returns the complex value in double.
template <typename T>
static __device__ cplx<double> mps_overlap(const EngineParams &P, const Smem<T> &S, int64_t shot, const Scratch<T> &X,
                                           const cplx<T> *phi, const int *phi_chi, bool with_op, int m) {
  const int n = P.n;
  const cplx<T> one = cmake<T>(1, 0), zero = cmake<T>(0, 0);
  MpoSpec<T> sp;
  sp.kind = MPO_ROT; sp.lo = -1; sp.hi = -1; sp.j = -1;
  sp.w0 = one; sp.w1 = one; sp.v0 = zero; sp.v1 = zero;
  for (int k = 0; k < n; ++k) {
    const cplx<T> *A = site_ptr<T>(P, shot, k);
    const int clm = S.chi[k], crm = S.chi[k + 1];
    const int clp = phi_chi[k], crp = phi_chi[k + 1];
    const cplx<T> *B = phi + P.site_off[k];
    const bool acts = with_op && (((S.ppx[k >> 6] | S.ppz[k >> 6]) >> (k & 63)) & 1);
    if (acts) {
      cplx<T> op[4];
      site_op(sp, S.ppx, S.ppz, k, 1, op);
      const int64_t tot = static_cast<int64_t>(clp) * 2 * crp;
      for (int64_t e = tid(); e < tot; e += kThreads) {
        const int r = static_cast<int>(e % crp), s2 = static_cast<int>((e / crp) % 2);
        const int64_t l = e / (2 * crp);
        cplx<T> v = zero;
        cfma(v, op[s2 * 2 + 0], B[(l * 2 + 0) * crp + r]);
        cfma(v, op[s2 * 2 + 1], B[(l * 2 + 1) * crp + r]);
        X.sa[e] = v;
      }
      __syncthreads();
      B = X.sa;
    }
    if (k == 0) {  // E = A_mu^dag B over the physical index (chi_0 = 1)
      cgemm<T, 1, 0>(crm, crp, 2 * clm, one, A, crm, B, crp, zero, X.e, crp, S.tile);
    } else {
      cgemm<T, 0, 0>(clm, 2 * crp, clp, one, X.e, clp, B, 2 * crp, zero, X.te, 2 * crp, S.tile);
      cgemm<T, 1, 0>(crm, crp, 2 * clm, one, A, crm, X.te, crp, zero, X.e, crp, S.tile);
    }
  }
  const cplx<T> v = X.e[0];
  cplx<double> r = cmake<double>(static_cast<double>(v.re), static_cast<double>(v.im));
  const cplx<double> ph = ipow<double>(m);
  r = cmul(ph, r);
  __syncthreads();
  return r;
}

// Backward pass of the adjoint (see stn_logprob_grad): one CTA per record,
// the shot's MPS holding mu (initially the final state of the forced forward
// pass), the ops walked from last to first.  At a rotation of pair k the term
// 2 Re <mu| (-i P') |phi_j> / <mu|phi_j> is added to grad[k] (phi_j the
// stored state after that rotation), then mu <- exp(+i theta P') mu; a case-A
// measurement applies its projector again, a case-B measurement applies
// U |v><0|_j; every application is followed by the truncating sweep.
// Clifford gates and Paulis only changed the frame and leave mu alone.
template <typename T>
__global__ void __launch_bounds__(kThreads, kLight ? 2 : 1) adjoint_kernel(EngineParams P, double *grad) {
  extern __shared__ __align__(16) char smem_raw[];
  tc_disable();
  const int n = P.n, W = P.W;
  Smem<T> S = carve<T>(smem_raw, n, W, P.svd_elems);
  Scratch<T> X = scratch_for<T>(P, P.work_c);
  for (int64_t shot = blockIdx.x; shot < P.shots; shot += gridDim.x) {
    for (int e = tid(); e <= n; e += kThreads) S.chi[e] = P.chi[shot * (n + 1) + e];
    if (tid() == 0) {
      S.misc[M_CENTER] = P.center[shot];
      S.misc[M_FAIL] = P.status[shot];
      S.misc[M_MAXCHI] = P.maxchi[shot];
      S.dmisc[D_DISC] = 0.0;
      tally(S.dmisc, D_FLOPS) = 0;
    }
    __syncthreads();
    for (int oi = P.n_ops_total - 1; oi >= 0 && !S.misc[M_FAIL]; --oi) {
      const Op op = P.ops[oi];
      if (op.kind != OP_ROT && op.kind != OP_MEAS) continue;
      const int64_t t = shot * P.n_ops_total + oi;
      const int32_t *ti = P.tape_info + t * kTapeInts;
      const int info = ti[0], lo = ti[1], hi = ti[2], jq = ti[3];
      const int m = info & 3;
      if (tid() < W) {
        S.ppx[tid()] = P.tape_px[t * W + tid()];
        S.ppz[tid()] = P.tape_pz[t * W + tid()];
      }
      __syncthreads();
      MpoSpec<T> &sp = *S.spec;
      if (op.kind == OP_ROT) {
        const int64_t slot = shot * P.n_rot + P.rot_ord[oi];
        const cplx<T> *phi = reinterpret_cast<const cplx<T> *>(P.phi_store) + slot * P.slab_elems;
        const int *phi_chi = P.phi_chi + slot * (n + 1);
        const cplx<double> num = mps_overlap<T>(P, S, shot, X, phi, phi_chi, true, m + 3);  // (-i) i^m
        const cplx<double> den = mps_overlap<T>(P, S, shot, X, phi, phi_chi, false, 0);
        if (tid() == 0) {
          const double d2 = den.re * den.re + den.im * den.im;
          const double re = (num.re * den.re + num.im * den.im) / d2;  // Re(num / den)
          if (!(d2 > 0.0) || !isfinite(re)) S.misc[M_FAIL] = STN_ENUMERIC;
          else atomicAdd(&grad[op.idx], 2.0 * re);
          const double th = P.theta[op.idx];
          sp.kind = MPO_ROT;
          sp.lo = lo; sp.hi = hi; sp.j = -1;
          sp.w0 = cmake<T>(static_cast<T>(cos(th)), 0);
          sp.w1 = cmul(cmake<T>(0, static_cast<T>(sin(th))), ipow<T>(m));  // +i sin(theta) i^m
        }
      } else if (tid() == 0) {
        const int caseB = (info >> 2) & 1, bit = (info >> 3) & 1, lidx = (info >> 4) & 3, neg = (info >> 6) & 1;
        sp.lo = lo; sp.hi = hi; sp.j = jq;
        sp.w0 = cmake<T>(1, 0);
        sp.w1 = cmake<T>(1, 0);
        if (!caseB) {  // the forward projector (I + (-1)^b P')/2 again
          const int sgn = (bit ? -1 : 1) * ((m & 2) ? -1 : 1);
          sp.kind = MPO_PROJ_Z;
          sp.par = sgn > 0 ? 0 : 1;
        } else {  // U |v><0|_j, v the lambda eigenvector of the site-j letter
          (void)neg;
          const T r2 = static_cast<T>(0.70710678118654752440);
          const bool zj = lidx >= 2;
          const bool lam_neg = lidx & 1;
          sp.kind = MPO_ADJ_B;
          sp.v0 = cmake<T>(r2, 0);
          sp.v1 = zj ? cmake<T>(0, lam_neg ? -r2 : r2) : cmake<T>(lam_neg ? -r2 : r2, 0);
        }
      }
      __syncthreads();
      if (S.misc[M_FAIL]) break;
      const int c0 = S.misc[M_CENTER];
      const int tgt = c0 < lo ? lo : (c0 > hi ? hi : c0);
      if (tgt != c0) mps_move_center<T>(P, S, shot, X, tgt);
      if (S.misc[M_FAIL]) break;
      mps_prepare<T>(P, S, shot, X, lo, hi, false);
      __syncthreads();
      mps_finish<T>(P, S, shot, X, lo, hi);
      __syncthreads();
    }
    for (int e = tid(); e <= n; e += kThreads) P.chi[shot * (n + 1) + e] = S.chi[e];
    if (tid() == 0) {
      P.center[shot] = S.misc[M_CENTER];
      P.status[shot] = S.misc[M_FAIL];
      if (S.misc[M_FAIL]) atomicCAS(P.err, 0, S.misc[M_FAIL]);
    }
    __syncthreads();
  }
}

template <typename T>
cudaError_t launch_adjoint_t(const EngineParams &p, double *grad, int grid, cudaStream_t s) {
  size_t smem = smem_bytes<T>(p.n, p.W, p.svd_elems);
  cudaError_t e = cudaFuncSetAttribute(adjoint_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  adjoint_kernel<T><<<grid, kThreads, smem, s>>>(p, grad);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_diag_t(const EngineParams &p, int what, int target, int cut, const int32_t *lq, int nl,
                          int letter, double *out, int *count, int grid, cudaStream_t s) {
  size_t smem = smem_bytes<T>(p.n, p.W, p.svd_elems);
  cudaError_t e = cudaFuncSetAttribute(diag_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  diag_kernel<T><<<grid, kThreads, smem, s>>>(p, what, target, cut, lq, nl, letter, out, count);
  return cudaGetLastError();
}

template <typename T, int B>
cudaError_t launch_round_b(const EngineParams &p, int grid, cudaStream_t s) {
  size_t smem = smem_bytes<T>(p.n, p.W, p.svd_elems);
  cudaError_t e = cudaFuncSetAttribute(round_kernel<T, B>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  round_kernel<T, B><<<grid, kThreads, smem, s>>>(p);
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_round_t(const EngineParams &p, int grid, int sms, cudaStream_t s) {
  if constexpr (kLight) {
    if (grid > sms) return launch_round_b<T, 2>(p, grid, s);
  }
  return launch_round_b<T, 1>(p, grid, s);
}

STN_END
