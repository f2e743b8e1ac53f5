// Building blocks of the exact-split (Ozaki) matrix products on the tensor cores: PTX wrappers,
// bounded waits, float <-> fixed point, the digit planes, and the issue of one K stage's MMAs.
//
// A product of a float64 row x with a fixed matrix B is made exact up to the rounding of the two
// operands: x becomes the integers X_k = round(x_k 2^(62-E)) (|x_k| < 0.98 2^E over the row), B
// the integers Y_nk = round(B_nk 2^q), |Y| <= 2^54, written with eight and seven signed base-256
// digits,
//   X_k = sum_{i=0..7} a_ik 256^(7-i),  a_ik in [-128, 127],
// which bf16 holds exactly.  A digit product sum_k a_ik b_jnk is an integer, and the products with
// the same i + j = d share one fp32 accumulator G_d: |G_d| <= 7 2^14 K < 2^24 for K <= 144, so
// every accumulation is exact.  d <= 7 is kept (35 products), and
//   sum_k X_k Y_nk = 256^7 U,  U = sum_{d<=6} 256^(6-d) G_d + G_7 / 256
// is recombined in 64-bit integers; transforms with longer sums are cut into K groups of at most 144
// whose recombined integers are added.
//
// The error against exact sums (rows of decaying coefficients, transforms of 96 x 96 x 65 fields): the
// eighth digit of X takes the rounding of the small elements of a row, 2^-55 of its largest in seven
// digits, out of the result, and the eighth diagonal the dropped products, which with seven (28
// products) are 2^-51 of max|x| max|B|.  With seven digits and 28 (z) and 34 (x, y) products a backward
// transform was four times less accurate than by FFT (7.8e-16 against 1.9e-16 of the field).
//
// The seven B digit planes of an output slice are stacked into one 7 NT-row operand, so A plane i
// needs one MMA chain over rows 0 .. (8-i) NT (at most 7 NT) with its accumulator at column i NT:
// product (i, j) lands on diagonal i + j.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "ch_common.cuh"

namespace chf {
namespace tc {

constexpr int kRows = 128;        // rows per tile = tensor-memory lanes
constexpr int kPlanes = 7;        // base-256 digits of a matrix element
constexpr int kAPlanes = 8;       // and of a row's element
constexpr int kDiags = 8;         // accumulators (diagonals of digit products)
constexpr int kKS = 16;           // K per pipeline stage (one MMA k-step)
constexpr int kMaxK = 144;        // K up to which the fp32 accumulators stay exact
constexpr int kNTMax = 64;        // columns of an output slice (8 x 64 tensor-memory columns)
constexpr int kPlaneBytes = kRows * kKS * 2;             // one A digit plane of a stage
constexpr int kABytes = kAPlanes * kPlaneBytes;           // the A planes of a stage
constexpr uint32_t kALbo = kRows * 16;                   // A: bytes between 8-element K groups
__host__ __device__ constexpr int b_stage_bytes(int NT) { return kPlanes * NT * kKS * 2; }
constexpr unsigned long long kBias = 0x0080808080808080ull;   // 128 sum_{t<7} 256^t
constexpr unsigned long long kABias = 0x8080808080808080ull;  // 128 sum_{t<8} 256^t
constexpr uint64_t kWaitNs = 1000000000ull;                   // bound of every device wait

// ---- PTX wrappers -----------------------------------------------------------------------------
__device__ __forceinline__ uint32_t su32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// shared-memory matrix descriptor, no swizzle: lbo = byte stride between core matrices along K,
// sbo = byte stride between 8-row core-matrix groups along M (or N); version 1 at bit 46
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}
__device__ __forceinline__ uint64_t gtime() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// bounded wait for the phase with the given parity; false if it did not complete in time
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.b32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// wait for the phase with the given parity until the global timer passes `deadline`
__device__ __forceinline__ bool mbar_wait_until(uint32_t bar, uint32_t parity,
                                                uint64_t deadline) {
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (gtime() > deadline) return false;
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_try(bar, parity)) return true;   // the common case: no clock read
  return mbar_wait_until(bar, parity, gtime() + kWaitNs);
}
// The waits of one thread.  The first wait that runs out clears `ok`; every later wait returns
// false at once, so a thread spends at most one bound waiting in vain however many waits follow
// (the transform kernels' warps then leave their loops, the issuer after draining its MMAs).
struct Waiter {
  bool ok = true;
  __device__ __forceinline__ bool wait(uint32_t bar, uint32_t parity) {
    ok = ok && mbar_wait(bar, parity);
    return ok;
  }
  // the same for a whole warp: false for all lanes if it ran out for any
  __device__ __forceinline__ bool wait_warp(uint32_t bar, uint32_t parity) {
    ok = __all_sync(0xffffffffu, ok && mbar_wait(bar, parity)) != 0;
    return ok;
  }
};
__device__ __forceinline__ void mma_bf16(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                         uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
// L2 policy that keeps lines resident (the matrix digits, re-read by every tile) ahead of
// the streamed rows and outputs
__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// bulk copy global -> shared with completion on an mbarrier, read under the L2 policy `pol`
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar, uint64_t pol) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
      "[%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(pol)
      : "memory");
}
// 4-column loads (one per diagonal accumulator, `stride` columns apart) of this warp's 32 lanes,
// then one wait that the values depend on.  The loads are .aligned: every lane of the warp executes
// them together, so the warp is brought together here, after whatever its lanes did apart (the
// stores of a ragged last tile, whose rows only some lanes have).
__device__ __forceinline__ void tmem_ldx4(uint32_t addr, int stride, uint32_t (&v)[kDiags][4]) {
  __syncwarp();
#pragma unroll
  for (int d = 0; d < kDiags; ++d)
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[d][0]), "=r"(v[d][1]), "=r"(v[d][2]), "=r"(v[d][3])
                 : "r"(addr + (uint32_t)(d * stride)));
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0][0]), "+r"(v[0][1]), "+r"(v[0][2]), "+r"(v[0][3]), "+r"(v[1][0]),
                 "+r"(v[1][1]), "+r"(v[1][2]), "+r"(v[1][3]), "+r"(v[2][0]), "+r"(v[2][1]),
                 "+r"(v[2][2]), "+r"(v[2][3]), "+r"(v[3][0]), "+r"(v[3][1]), "+r"(v[3][2]),
                 "+r"(v[3][3]), "+r"(v[4][0]), "+r"(v[4][1]), "+r"(v[4][2]), "+r"(v[4][3]),
                 "+r"(v[5][0]), "+r"(v[5][1]), "+r"(v[5][2]), "+r"(v[5][3]), "+r"(v[6][0]),
                 "+r"(v[6][1]), "+r"(v[6][2]), "+r"(v[6][3]), "+r"(v[7][0]),
                 "+r"(v[7][1]), "+r"(v[7][2]), "+r"(v[7][3])
               :
               : "memory");
}

// ---- float <-> fixed point --------------------------------------------------------------------
// Storage types of a row's elements: the bit pattern, its magnitude bits (an unsigned key that
// orders |x|; infinities and NaNs are the largest) and the exponent field of the row scale.
// maxe = row_scale(largest key) is the exponent field of the row's largest element, plus one when
// that element is above 0.975 of the next power of two: |x| < 0.976 2^E with E = maxe - EOFF, so
// the sum or difference of two elements stays inside the eight signed base-256 digits (0.996 2^63).
template <typename T> struct FBits;
template <> struct FBits<double> {
  static constexpr int EMAX = 0x7FF, EOFF = 1022, KEY_MB = 20;
  typedef unsigned long long U;
  __device__ static U bits(double x) { return (U)__double_as_longlong(x); }
  // (the low word only tells the smallest subnormals from zero)
  __device__ static unsigned key(U b) {
    return max((unsigned)(b >> 32) & 0x7FFFFFFFu, (unsigned)((unsigned)b != 0));
  }
};
template <> struct FBits<float> {
  static constexpr int EMAX = 0xFF, EOFF = 126, KEY_MB = 23;
  typedef unsigned int U;
  __device__ static U bits(float x) { return __float_as_uint(x); }
  __device__ static unsigned key(U b) { return b & 0x7FFFFFFFu; }
};
// double-float h + l: the bits of h in the low word, of l in the high word; the row scale comes
// from h (|l| <= ulp(h) / 2)
template <> struct FBits<df> {
  static constexpr int EMAX = 0xFF, EOFF = 126, KEY_MB = 23;
  typedef unsigned long long U;
  __device__ static U bits(df x) {
    return (U)__float_as_uint(x.h) | ((U)__float_as_uint(x.l) << 32);
  }
  __device__ static unsigned key(U b) { return (unsigned)b & 0x7FFFFFFFu; }
};
// A row of zeros takes the scale kTinyScale.
constexpr int kNanRow = 1 << 14;   // scale of a row that holds an infinity or NaN
constexpr int kTinyScale = 64;     // row scales below it need care with subnormals (Fixed)
template <typename T> __device__ __forceinline__ int row_scale(unsigned key) {
  typedef FBits<T> F;
  const int e = (int)(key >> F::KEY_MB);
  if (e >= F::EMAX) return kNanRow;
  if (key == 0) return kTinyScale;
  const unsigned frac = key & ((1u << F::KEY_MB) - 1u);
  return max(e, 1) + (frac > (unsigned)(0.95 * (1 << F::KEY_MB)) ? 1 : 0);
}

// round(x 2^(62-E)) of the element with bit pattern b in a row of scale maxe (E = maxe - EOFF);
// zero in a row that holds an infinity or NaN (kNanRow), whose results are NaN.  TINY = false: the
// implicit mantissa bit is set whatever the exponent field, which is right for normal numbers and
// harmless for zeros and subnormals once the row scale is at least kTinyScale (they shift out).
template <bool TINY> __device__ __forceinline__ long long fixed_f32(unsigned b, int maxe) {
  int ef = (int)((b >> 23) & 0xFFu);
  unsigned m = (b & 0x7FFFFFu) | 0x800000u;
  if (TINY && ef == 0) {
    m = b & 0x7FFFFFu;
    ef = 1;
  }
  const int sh = min(maxe - ef, 63);
  const unsigned long long r = (((unsigned long long)m << 39 >> sh) + 1ull) >> 1;
  const long long s = (long long)((int)b >> 31);
  return ((long long)r ^ s) - s;
}
template <typename T, bool TINY> struct Fixed;
template <bool TINY> struct Fixed<double, TINY> {
  __device__ __forceinline__ static long long of(unsigned long long b, int maxe) {
    const unsigned hi = (unsigned)(b >> 32);
    int ef = (int)((hi >> 20) & 0x7FFu);
    unsigned mh = (hi & 0xFFFFFu) | 0x100000u;
    if (TINY && ef == 0) {
      mh = hi & 0xFFFFFu;
      ef = 1;
    }
    const int sh = min(maxe - ef, 63);
    const unsigned long long m = (((unsigned long long)mh << 32) | (unsigned)b) << 10;
    const unsigned long long r = ((m >> sh) + 1ull) >> 1;
    const long long s = (long long)((int)hi >> 31);
    return ((long long)r ^ s) - s;
  }
};
template <bool TINY> struct Fixed<float, TINY> {
  __device__ __forceinline__ static long long of(unsigned b, int maxe) {
    return fixed_f32<TINY>(b, maxe);
  }
};
// double-float: both parts converted and added (one extra unit of rounding at most)
template <bool TINY> struct Fixed<df, TINY> {
  __device__ __forceinline__ static long long of(unsigned long long b, int maxe) {
    return fixed_f32<TINY>((unsigned)b, maxe) + fixed_f32<true>((unsigned)(b >> 32), maxe);
  }
};

// Digit plane i (0 = most significant) of two values, as two bf16 in one word (first in the low
// half): byte 7 - i of the biased integers, u, stands for the digit u - 128.  With l = u mod 128,
// the bf16 128 + l is 0x4300 | l, and the digit is (128 + l) - 256 or (128 + l) - 128 (bit 7 of u
// clear or set; the bf16 -256 and -128 differ in exactly that bit of 0xC380), one exact bf16 add.
__device__ __forceinline__ uint32_t digit_pair(uint32_t w0, uint32_t w1, int byte) {
  const uint32_t w = __byte_perm(w0, w1, (uint32_t)(byte | (byte << 4) | ((4 + byte) << 8) |
                                                    ((4 + byte) << 12)));
  const uint32_t a = (w & 0x007F007Fu) | 0x43004300u;
  const uint32_t c = (w & 0x00800080u) ^ 0xC380C380u;
  __nv_bfloat162 r = __hadd2(*reinterpret_cast<const __nv_bfloat162*>(&a),
                             *reinterpret_cast<const __nv_bfloat162*>(&c));
  return *reinterpret_cast<uint32_t*>(&r);
}

// the high and low words of biased fixed-point values, added apart
struct WordSums {
  unsigned long long h = 0, l = 0;
  __device__ __forceinline__ void add(unsigned long long v) {
    h += (unsigned)(v >> 32);
    l += (unsigned)v;
  }
  // the sums of the values without their bias, of n values: h 2^32 + l
  __device__ __forceinline__ long long high(int n) const {
    return (long long)(h - (unsigned long long)n * (unsigned)(kABias >> 32));
  }
  __device__ __forceinline__ long long low(int n) const {
    return (long long)(l - (unsigned long long)n * (unsigned)kABias);
  }
};
// such a sum times 2^e, rounded once (both words are below 2^53, so their conversions are exact)
template <typename TO> __device__ TO words_scaled(long long h, long long l, int e);
template <> __device__ __forceinline__ double words_scaled<double>(long long h, long long l, int e) {
  return ldexp(fma(__ll2double_rn(h), 4294967296.0, __ll2double_rn(l)), e);
}
template <> __device__ __forceinline__ float words_scaled<float>(long long h, long long l, int e) {
  return (float)words_scaled<double>(h, l, e);
}
template <> __device__ __forceinline__ df words_scaled<df>(long long h, long long l, int e) {
  const double v = words_scaled<double>(h, l, e);
  const float hi = (float)v;
  return df(hi, (float)(v - (double)hi));
}

// round(U / 64) of column e of the diagonal accumulators (exact integers below 2^24 held as
// fp32), U = sum_d 256^(6-d) G_d.  Sums are formed modulo 2^64; |U| / 64 < 2^63 for sums of at most
// 496 terms per row (|sum_k x_k B_nk| < 496 max|x| max|B|).  The first NMAG accumulators are known
// to stay within 2^22 and convert by one float addition (the low bits of 1.5 2^23 + G are G), the
// others by the conversion instruction (a quarter of the rate).
template <int NMAG>
__device__ __forceinline__ long long recombine(const uint32_t (&v)[kDiags][4], int e) {
  int g[kDiags];
#pragma unroll
  for (int d = 0; d < kDiags; ++d)
    g[d] = d < NMAG ? __float_as_int(__uint_as_float(v[d][e]) + 12582912.0f) - 0x4B400000
                    : __float2int_rz(__uint_as_float(v[d][e]));
  // h, m (and q, when every |G| <= 2^22) fit 32 bits; G_4 256^2 + G_5 256 = 2^8 q and
  // G_6 256 + G_7 = r contribute 4 q + round(r / 2^14) to U / 64
  const int h = g[0] * 256 + g[1], m = g[2] * 256 + g[3];
  long long l;
  if (NMAG == kDiags) {
    const int q = g[4] * 256 + g[5];
    const int r = (g[6] * 256 + g[7] + 8192) >> 14;
    l = (long long)q * 4 + (long long)r;
  } else {
    l = (long long)g[4] * 1024 + ((long long)g[5] * 4 +
        (((long long)g[6] * 256 + (long long)g[7] + 8192) >> 14));
  }
  return (long long)((unsigned long long)(unsigned)h << 34) + ((long long)m * 262144 + l);
}

// T 2^e rounded once to the output type: the integer converts in one instruction and the power of
// two is added to the exponent field, right when safe_exp(e) (the result of every |T| in
// 1 .. 2^63 is a normal number).
template <typename TO> __device__ __forceinline__ bool safe_exp(int e) {
  return FBits<TO>::EMAX == 0xFF ? e > -120 && e < 60 : e > -1000 && e < 950;
}
template <typename TO> __device__ TO scaled(long long T, int e);
template <> __device__ __forceinline__ double scaled<double>(long long T, int e) {
  const double v = __ll2double_rn(T);
  return __hiloint2double(__double2hiint(v) + (T != 0 ? e << 20 : 0), __double2loint(v));
}
// the same to nearest even by integer operations alone: the conversion instruction runs on the
// float64 pipe (1.9 a clock per SM), so the epilogues send every second value this way
template <typename TO> __device__ __forceinline__ TO scaled_alu(long long T, int e) {
  return scaled<TO>(T, e);
}
template <> __device__ __forceinline__ double scaled_alu<double>(long long T, int e) {
  const int sg = (int)(T >> 63);
  const unsigned long long a = ((unsigned long long)T ^ (unsigned long long)(long long)sg) -
                               (unsigned long long)(long long)sg;   // |T| < 2^63
  const int lz = __clzll((long long)a);
  const unsigned long long n = a << (lz - 1);                // leading one at bit 62
  const unsigned long long m = (n + 0x1FFull + ((n >> 10) & 1ull)) >> 10;   // 53 bits, or 2^53
  const int hi = (int)(m >> 32) + ((1085 - lz + e) << 20);   // m carries the implicit bit
  return __hiloint2double((T != 0 ? hi : 0) | (sg & (int)0x80000000), T != 0 ? (int)m : 0);
}
template <> __device__ __forceinline__ float scaled<float>(long long T, int e) {
  return __int_as_float(__float_as_int(__ll2float_rn(T)) + (T != 0 ? e << 23 : 0));
}
// double-float result: the high part rounded to float, the low part from the exact remainder
template <> __device__ __forceinline__ df scaled<df>(long long T, int e) {
  const long long hi = __float2ll_rn(__ll2float_rn(T));   // |T| < 2^62.93: no overflow
  return df(scaled<float>(hi, e), scaled<float>(T - hi, e));
}
// the same outside the safe exponents
template <typename TO> __device__ TO scaled_any(long long T, int e);
template <> __device__ __forceinline__ double scaled_any<double>(long long T, int e) {
  return ldexp(__ll2double_rn(T), e);
}
template <> __device__ __forceinline__ float scaled_any<float>(long long T, int e) {
  return ldexpf(__ll2float_rn(T), e);
}
template <> __device__ __forceinline__ df scaled_any<df>(long long T, int e) {
  const long long hi = __float2ll_rn(__ll2float_rn(T));
  return df(ldexpf(__ll2float_rn(hi), e), ldexpf(__ll2float_rn(T - hi), e));
}
template <typename TO> __device__ __forceinline__ TO qnan();
template <> __device__ __forceinline__ double qnan<double>() {
  return __longlong_as_double(0x7FF8000000000000ll);
}
template <> __device__ __forceinline__ float qnan<float>() { return __uint_as_float(0x7FC00000u); }
template <> __device__ __forceinline__ df qnan<df>() {
  return df(__uint_as_float(0x7FC00000u), __uint_as_float(0x7FC00000u));
}

// ---- one K stage's MMAs -----------------------------------------------------------------------
// A planes at shared address sA, the stacked B planes (7 NT rows) at sB, both 16 K wide in the
// canonical no-swizzle K-major core-matrix layout; accumulators from tensor-memory column tmem.
// A plane i times B rows 0 .. min(7, 8-i) NT, in pieces of at most 256 columns of equal width (an MMA of
// M = 128 takes N / 2 cycles, but not less than about 50).  init: the accumulators start from zero
// (plane 0 covers all their columns).  NT is a template argument because the single issuing thread
// is what limits the rate otherwise (NT = 64: 28 products took 912 cycles of MMAs per stage;
// with the pieces worked out at run time the issue took 2040).
template <int NT>
__device__ __forceinline__ void issue_stage_nt(uint32_t tmem, uint32_t sA, uint32_t sB, bool init) {
  // bf16 x bf16 -> fp32, both K-major, M = 128 (N added per MMA)
  constexpr uint32_t idesc0 =
      (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kRows >> 4) << 24);
  const uint64_t a0 = sdesc(sA, kALbo, 128), b0 = sdesc(sB, (uint32_t)(kPlanes * NT * 16), 128);
#pragma unroll
  for (int i = 0; i < kAPlanes; ++i) {
    // diagonals i .. 6, and diagonal 7 of planes 1 .. 7; plane 1 touches diagonal 7 first, in an MMA
    // of its own that may start it from zero
    const int nb = i > 1 ? kDiags - i : kPlanes - i;
    const int ntot = nb * NT, np = (ntot + 255) / 256;
    const int len = (ntot / np + 15) / 16 * 16;
#pragma unroll
    for (int n0 = 0; n0 < ntot; n0 += len) {
      const int nlen = len < ntot - n0 ? len : ntot - n0;
      mma_bf16(tmem + (uint32_t)(i * NT + n0), a0 + (uint64_t)(i * (kPlaneBytes / 16)),
               b0 + (uint64_t)n0, idesc0 | ((uint32_t)(nlen >> 3) << 17),
               (uint32_t)!(init && i == 0));
    }
    if (i == 1)
      mma_bf16(tmem + (uint32_t)(7 * NT), a0 + (uint64_t)(kPlaneBytes / 16),
               b0 + (uint64_t)(6 * NT), idesc0 | ((uint32_t)(NT >> 3) << 17), (uint32_t)!init);
  }
}
__device__ __forceinline__ void issue_stage(uint32_t tmem, uint32_t sA, uint32_t sB, int NT,
                                            bool init) {
  switch (NT) {
    case 16: issue_stage_nt<16>(tmem, sA, sB, init); break;
    case 32: issue_stage_nt<32>(tmem, sA, sB, init); break;
    case 48: issue_stage_nt<48>(tmem, sA, sB, init); break;
    default: issue_stage_nt<64>(tmem, sA, sB, init); break;
  }
}

}  // namespace tc
}  // namespace chf
