// Division and square root of binary64 on the FP32 and integer pipes.
//
// This part's FP64 pipe takes 2 instructions per clock per SM, its FP32 and
// integer pipes 128 and 64.  An IEEE FP64 division or square root as the
// compiler expands it holds the FP64 pipe for as long as 7.5 additions (143
// clocks a warp on one SM, measured by a throughput probe: 152 x 4 blocks of
// 256 threads, 4 chains a thread).  The forms here use no FP64 instruction:
//   * the FP32 reciprocal (reciprocal square root) of the operand's leading
//     24 bits, and two Newton steps whose residuals run over the whole operand
//     in FP32 fused multiply-adds, give 45 bits;
//   * put together as an integer significand, the quotient's (root's) exact
//     remainder follows from the low 64 bits of an integer product (it is
//     small, so the high bits are known to cancel);
//   * remainder times reciprocal in FP32 (below 2^9, off by less than 2^-13),
//     rounded to the nearest integer, is the last correction.  Where it lies
//     within 2^-12 of the middle of two integers the rounding is decided by
//     an exact integer comparison.
// So every result is the correctly rounded one, bit for bit what the IEEE
// operation returns, which the tests compare on hard operands.  (Newton's
// iteration and exact remainders: Markstein, IBM J. Res. Dev. 34 (1990) 111.)
//
// Operands: what div_by, rcp_by, sqrt_ranged and mul_int need is normal
// operands (a numerator or a second factor also zero) and a normal result:
// their exponents are sums and differences in one integer word, without a
// check.  The range tests (F64Range) bound the operands they see by 2^-400 ..
// 2^400, so that a few may be combined before the next test; the longest chain,
// the reciprocal of c^2 = gamma p / rho through its root (gamma within 2^+-100,
// p and rho tested), stays within 2^+-905.  A
// caller collects the tests and repeats its whole evaluation with plain
// products or IEEE operations when one fails, or uses the checked forms
// (div_f64, sqrt_f64), which take the IEEE operation for such an operand.
// NaN, infinities, subnormals, zero denominators and negative radicands fail
// the test.
#pragma once
#include <cuda_runtime.h>

namespace cgk {

constexpr unsigned kF64Lo = (1023u - 400u) << 20;  // high word of 2^-400
constexpr unsigned kF64Span = 800u << 20;          // up to (not including) 2^400

// The range tests of several operands, collected: ok() holds when every
// operand seen was in range.
struct F64Range {
  unsigned worst = 0u;
  __device__ __forceinline__ void see(unsigned t) { worst = t > worst ? t : worst; }
  // a positive operand
  __device__ __forceinline__ void pos(double x) { see((unsigned)__double2hiint(x) - kF64Lo); }
  // an operand of either sign
  __device__ __forceinline__ void any(double x) { see(((unsigned)__double2hiint(x) & 0x7fffffffu) - kF64Lo); }
  // an operand of either sign, or zero
  __device__ __forceinline__ void any0(double x) {
    const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu;
    see((h | (unsigned)__double2loint(x)) == 0u ? 0u : h - kF64Lo);
  }
  __device__ __forceinline__ bool ok() const { return worst < kF64Span; }
};

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ unsigned long long u64_of(unsigned hi, unsigned lo) {
  return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ unsigned hi_of(unsigned long long x) { return (unsigned)(x >> 32); }

// The part of the significand below its leading 24 bits in units of the last
// of them: its own leading 23 bits, and half a unit for the 6 that follow.
__device__ __forceinline__ float low_bits(unsigned lo) {
  return __fadd_rn(__uint_as_float(((lo >> 6) & 0x007fffffu) | 0x3f800000u), 0x1p-24f - 1.0f);
}

// The nearest integer to v (|v| < 2^22); near: v lies within 2^-12 of the
// middle of two integers.
__device__ __forceinline__ int nearest(float v, bool& near) {
  const float magic = 12582912.0f;  // 1.5 2^23
  const float t = __fadd_rn(v, magic);
  near = fabsf(__fsub_rn(v, __fsub_rn(t, magic))) > 0.5f - 0x1p-12f;
  return __float_as_int(t) - __float_as_int(magic);
}

// The divisor of one or more quotients: its significand B (53 bits), Y =
// 2^105 / B to a relative 2^-45, the FP32 reciprocal of B 2^-52, and the high
// word (exponent and sign).
struct Divisor {
  unsigned long long B, Y;
  float r;
  unsigned hi;
};

__device__ __forceinline__ Divisor divisor(double x) {
  Divisor D;
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  D.hi = hi & 0xfff00000u;
  D.B = u64_of((hi & 0x000fffffu) | 0x00100000u, lo);
  // |x| scaled to [1, 2): xh + xl 2^-23
  const float xh = __uint_as_float(__funnelshift_l(lo, (hi & 0x000fffffu) | 0x07f00000u, 3));
  const float xl = low_bits(lo);
  const float r0 = rcp_approx(xh), s = __fmul_rn(r0, 0x1p-23f);
  // r = 1/x rounded to 24 bits; e = 1 - x r, |e| < 2^-23
  const float r = __fmaf_rn(r0, __fmaf_rn(-xl, s, __fmaf_rn(-xh, r0, 1.0f)), r0);
  const float e = __fmaf_rn(-xl, s, __fmaf_rn(-xh, r, 1.0f));
  const float magic = 1.5f * 0x1p-23f;  // units of 2^-46
  const int units = __float_as_int(__fmaf_rn(r, e, magic)) - __float_as_int(magic);
  const unsigned b = __float_as_uint(r);  // r in [1/2, 1]
  D.Y = u64_of((b - 0x3e800000u) >> 3, b << 29) + (unsigned long long)((long long)units * 128);
  D.r = r;
  return D;
}

// Q0 + (N - Q0 B) / B rounded to the nearest integer, from the remainder R = N - Q0 B.
static __device__ __noinline__ int nearest_exact(long long R, unsigned long long B, int d) {
  const long long t = 2 * (R - (long long)d * (long long)B);
  return t > (long long)B ? d + 1 : (t < -(long long)B ? d - 1 : d);
}
__device__ __forceinline__ unsigned long long round_quotient(unsigned long long Q0, long long R, const Divisor& D) {
  bool near;
  int d = nearest(__fmul_rn(__int2float_rn((int)(R >> 32)), __fmul_rn(D.r, 0x1p-20f)), near);
  if (near) d = nearest_exact(R, D.B, d);
  return Q0 + (unsigned long long)(long long)d;
}

// a / x for the divisor D of x: a in range or zero.
__device__ __forceinline__ double div_by(double a, const Divisor& D) {
  const unsigned hi = (unsigned)__double2hiint(a), lo = (unsigned)__double2loint(a);
  const unsigned long long A = u64_of((hi & 0x000fffffu) | 0x00100000u, lo);
  // the quotient of the significands lies in (1/2, 2): scaled by 2^52, or by 2^53 if A < B
  const unsigned c = A < D.B ? 1u : 0u;
  const unsigned long long As = A << 11, Ys = D.Y << c;
  const unsigned a1 = hi_of(As), a0 = (unsigned)As, y1 = hi_of(Ys), y0 = (unsigned)Ys;
  const unsigned long long Q0 = (unsigned long long)a1 * y1 + __umulhi(a1, y0) + __umulhi(a0, y1);
  const long long R = (long long)(u64_of(lo << (20u + c), 0u) - Q0 * D.B);
  const unsigned long long Q = round_quotient(Q0, R, D);
  const unsigned rh = hi_of(Q) + (hi & 0xfff00000u) - D.hi + (1022u << 20) - (c << 20);
  const bool zero = ((hi & 0x7fffffffu) | lo) == 0u;
  return __hiloint2double((int)(zero ? (hi ^ D.hi) & 0x80000000u : rh), (int)(zero ? 0u : (unsigned)Q));
}

// 1 / x for the divisor D of x.
__device__ __forceinline__ double rcp_by(const Divisor& D) {
  // 2^105 / B, in (2^52, 2^53]
  const unsigned long long Q = round_quotient(D.Y, (long long)(0ull - D.Y * D.B), D);
  const unsigned rh = hi_of(Q) + (1022u << 20) + (1022u << 20) - D.hi;
  return __hiloint2double((int)rh, (int)(unsigned)Q);
}

static __device__ __noinline__ int nearest_root_exact(long long R, unsigned long long G, int d) {
  // (G + d + 1/2)^2 against G^2 + R: R - 2 G d - d^2 - (G + d) against 1/4, and the other side
  const long long Gd = (long long)G, t = R - 2 * Gd * d - (long long)d * d;
  return t > Gd + d ? d + 1 : (t < 1 - (Gd + d) ? d - 1 : d);
}

// sqrt(x), x positive and in range.
__device__ __forceinline__ double sqrt_ranged(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  // x = m 2^(2k), m in [1, 4): the leading 24 bits xh and the rest xl
  const unsigned hm = ((hi & 0x001fffffu) ^ 0x00100000u) + 0x07f00000u;  // high word of m, exponent bias 127
  const float xh = __uint_as_float(__funnelshift_l(lo, hm, 3));
  const float ulp = __uint_as_float((__float_as_uint(xh) & 0x7f800000u) - (23u << 23));
  const float xl = __fmul_rn(low_bits(lo), ulp);
  const float r = rsqrt_approx(xh);
  // g = sqrt(m) rounded to 24 bits (at least 1), c = (m - g^2) / (2 g)
  const float g0 = __fmul_rn(xh, r), h0 = __fmul_rn(0.5f, r);
  const float h = __fmaf_rn(h0, __fmaf_rn(-g0, r, 1.0f), h0);  // 1 / (2 g)
  const float g = fmaxf(__fmaf_rn(__fadd_rn(__fmaf_rn(-g0, g0, xh), xl), h, g0), 1.0f);
  const float c = __fadd_rn(__fmaf_rn(-g, g, xh), xl);
  const float magic = 1.5f * 0x1p-22f;  // units of 2^-45
  const int units = __float_as_int(__fmaf_rn(c, h, magic)) - __float_as_int(magic);
  const unsigned b = __float_as_uint(g);  // g in [1, 2]
  const unsigned long long G0 = u64_of((b - 0x3f000000u) >> 3, b << 29) + (unsigned long long)((long long)units * 128);
  // m 2^104 - G0^2
  const long long R = (long long)(u64_of(lo << (21u - ((hi >> 20) & 1u)), 0u) - G0 * G0);
  bool near;
  int d = nearest(__fmul_rn(__int2float_rn((int)(R >> 32)), __fmul_rn(h, 0x1p-20f)), near);
  if (near) d = nearest_root_exact(R, G0, d);
  const unsigned long long Q = G0 + (unsigned long long)(long long)d;
  const unsigned k = (unsigned)((int)((hi & 0x7ff00000u) - (hm & 0x7ff00000u) - (896u << 20)) >> 1);
  return __hiloint2double((int)(hi_of(Q) + (1022u << 20) + k), (int)(unsigned)Q);
}

// The divisor of a positive constant, on the host.
inline Divisor host_divisor(double x) {
  unsigned long long b;
  static_assert(sizeof b == sizeof x, "binary64");
  __builtin_memcpy(&b, &x, sizeof b);
  Divisor D;
  D.hi = (unsigned)(b >> 32) & 0xfff00000u;
  D.B = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  D.Y = (unsigned long long)(((unsigned __int128)1 << 105) / D.B);
  D.r = (float)(4503599627370496.0 / (double)D.B);
  return D;
}

// ---------------------------------------------------------------- products
// A correctly rounded product on the integer pipes: the 106-bit product of the
// significands in four 32 x 32 multiply-adds, normalised by at most one bit,
// rounded to nearest even on the bits below.  About 30 integer instructions,
// 18.9 clocks a warp on one SM where a DMUL is 18.7, but on other pipes: a
// loop of one addition and one product takes 18.7 clocks instead of 37.3 (the
// same probe).  So the products of an FP64-bound kernel are free as long as
// they are no more than its additions.
// a: in range; b: in range, or zero where ZB.
__device__ __forceinline__ unsigned long long mad_wide(unsigned a, unsigned b, unsigned long long c) {
  return (unsigned long long)a * b + c;
}
template <bool ZB>
__device__ __forceinline__ double mul_int(double a, double b) {
  const unsigned ah = (unsigned)__double2hiint(a), al = (unsigned)__double2loint(a);
  const unsigned bh = (unsigned)__double2hiint(b), bl = (unsigned)__double2loint(b);
  const unsigned a1 = __funnelshift_l(al, ah, 11) | 0x80000000u, a0 = al << 11;  // [2^63, 2^64)
  const unsigned b1 = (bh & 0x000fffffu) | 0x00100000u;                         // [2^52, 2^53)
  const unsigned long long t0 = mad_wide(a0, bl, 0ull), t1 = mad_wide(a1, bl, t0 >> 32),
                           t2 = mad_wide(a0, b1, (unsigned)t1);
  const unsigned long long H = mad_wide(a1, b1, t1 >> 32) + (t2 >> 32);  // [2^51, 2^53)
  const unsigned h1 = hi_of(H), h0 = (unsigned)H, l1 = (unsigned)t2, l0 = (unsigned)t0;
  const unsigned n = 1u - (h1 >> 20);
  const unsigned m1 = __funnelshift_l(h0, h1, n), m0 = __funnelshift_l(l1, h0, n);
  const unsigned low = l0 << n;
  const unsigned f = __funnelshift_l(l0, l1, n) | (low < 1u ? low : 1u);
  const unsigned long long M = u64_of(m1, m0) + (((unsigned long long)f + 0x7fffffffu + (m0 & 1u)) >> 32);
  const unsigned rh = hi_of(M) + (ah & 0xfff00000u) + (bh & 0xfff00000u) - (1023u << 20) - (n << 20);
  const bool zero = ZB && ((bh & 0x7fffffffu) | bl) == 0u;
  return __hiloint2double((int)(zero ? (ah ^ bh) & 0x80000000u : rh), (int)(zero ? 0u : (unsigned)M));
}

// Products of an evaluation that collects its range tests.  The additions of
// an evaluation hold the FP64 pipe anyway; a product with a factor that is
// known to be in range (a constant, a density) goes to the integer pipes (kk,
// kz), one of two unknown factors stays on the FP64 pipe (zz): testing two
// operands costs as much as the product, and with every product on the
// integer pipes the interface sweep is bound by its code size (instruction
// fetch) instead: 1.94 and 1.89 ms of MEG6 sweeps against 1.92 and 1.85.
struct F64Products {
  F64Range& R;
  static __device__ __forceinline__ double zz(double a, double b) { return a * b; }
  // a in range, b any (zero, or tested here)
  __device__ __forceinline__ double kz(double a, double b) const {
    R.any0(b);
    return mul_int<true>(a, b);
  }
  // both in range
  static __device__ __forceinline__ double kk(double a, double b) { return mul_int<false>(a, b); }
};
struct PlainProducts {
  template <typename T>
  static __device__ __forceinline__ T zz(T a, T b) { return a * b; }
  template <typename T>
  static __device__ __forceinline__ T kz(T a, T b) { return a * b; }
  template <typename T>
  static __device__ __forceinline__ T kk(T a, T b) { return a * b; }
};

// A factor used as known to be in range: tested with the rest.
__device__ __forceinline__ void require_range(const F64Products& P, double a) { P.R.any(a); }
template <typename T>
__device__ __forceinline__ void require_range(const PlainProducts&, T) {}

// Keeps a rare branch a branch: an FP64 instruction that is predicated off holds
// the pipe as long as one that runs (probe: a predicated DMUL beside a product
// on the integer pipes, 36.4 clocks; behind a call, 18.7), and the compiler
// predicates short branches that hold no call.
static __device__ __noinline__ void rare_branch() { asm volatile(""); }

// Where the additions are few beside the products and the loads, it takes less:
// us a pass of the triple point 1792 x 768 with plain and with integer-pipe
// products: Gaussian 431 and 276, interface LAD fluxes 334 and 216, E4 gradients
// 503 and 289, sensor 462 and 333.
//
// f(P) with the products of an FP64 evaluation on the integer pipes, and again
// with plain products where an operand was out of range (the same values
// otherwise); float: plain products.
template <typename T, class F>
__device__ __forceinline__ void with_products(F f) {
  if constexpr (sizeof(T) == 8) {
    F64Range R;
    f(F64Products{R});
    if (!R.ok()) {
      rare_branch();
      f(PlainProducts{});
    }
  } else {
    f(PlainProducts{});
  }
}

// ---------------------------------------------------------------- comparisons
// Comparisons of finite doubles on their bit patterns (a DSETP holds the FP64
// pipe as long as an addition does).
__device__ __forceinline__ long long bits64(double x) { return __double_as_longlong(x); }
__device__ __forceinline__ long long order_key(double x) {  // ordered like the doubles (and back again)
  const int hi = __double2hiint(x), s = hi >> 31;
  return (long long)u64_of((unsigned)(hi ^ (s & 0x7fffffff)), (unsigned)(__double2loint(x) ^ s));
}
__device__ __forceinline__ double from_key(long long k) {
  const int hi = (int)(k >> 32), s = hi >> 31;
  return __hiloint2double(hi ^ (s & 0x7fffffff), (int)(unsigned)k ^ s);
}
__device__ __forceinline__ long long kmin(long long a, long long b) { return a < b ? a : b; }
__device__ __forceinline__ long long kmax(long long a, long long b) { return a > b ? a : b; }
__device__ __forceinline__ double min_f64(double a, double b) { return order_key(a) < order_key(b) ? a : b; }
__device__ __forceinline__ double max_f64(double a, double b) { return order_key(a) > order_key(b) ? a : b; }
__device__ __forceinline__ bool is_nan(double x) {
  return ((unsigned long long)bits64(x) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull;
}
__device__ __forceinline__ bool is_nan(float x) { return (__float_as_uint(x) & 0x7fffffffu) > 0x7f800000u; }
// 0 <= x (either zero included, NaN not)
__device__ __forceinline__ bool nonneg(double x) {
  return (unsigned long long)bits64(x) <= 0x7ff0000000000000ull ||
         (__double2hiint(x) == (int)0x80000000 && __double2loint(x) == 0);
}
// the one of smaller magnitude where the signs agree, else zero
__device__ __forceinline__ double minmod_f64(double a, double b) {
  const bool same = (__double2hiint(a) ^ __double2hiint(b)) >= 0;
  const double m = (unsigned long long)bits64(a) < (unsigned long long)bits64(b) ? a : b;
  return same ? m : 0.0;
}
// x 2^K for normal x and result: an add to the exponent
template <int K>
__device__ __forceinline__ double scale2(double x) {
  return __hiloint2double(__double2hiint(x) + K * 0x00100000, __double2loint(x));
}
// x with its sign flipped where s (+1 or -1) is negative: s x
__device__ __forceinline__ double by_sign(double s, double x) {
  return __hiloint2double(__double2hiint(x) ^ (__double2hiint(s) & (int)0x80000000), __double2loint(x));
}

static __device__ __noinline__ double div_ieee(double a, double b) { return a / b; }
static __device__ __noinline__ double sqrt_ieee(double x) { return sqrt(x); }

// Checked forms: any operands.
__device__ __forceinline__ double div_f64(double a, double b) {
  F64Range R;
  R.any0(a);
  R.any(b);
  if (R.ok()) return div_by(a, divisor(b));
  return div_ieee(a, b);
}
__device__ __forceinline__ double sqrt_f64(double x) {
  F64Range R;
  R.pos(x);
  if (R.ok()) return sqrt_ranged(x);
  if ((__double2hiint(x) | __double2loint(x)) == 0) return x;  // +0
  return sqrt_ieee(x);
}

// ---------------------------------------------------------------- by type
// The forms above for double; for float (the mixed form) the plain operations.
__device__ __forceinline__ double div_t(double a, double b) { return div_f64(a, b); }
__device__ __forceinline__ float div_t(float a, float b) { return a / b; }
__device__ __forceinline__ double sqrt_t(double x) { return sqrt_f64(x); }
__device__ __forceinline__ float sqrt_t(float x) { return sqrtf(x); }
// 1/x
__device__ __forceinline__ double rcp_f64(double x) {
  F64Range R;
  R.any(x);
  return R.ok() ? rcp_by(divisor(x)) : div_ieee(1.0, x);
}
// m, or a where it is larger (m not negative, a not negative or NaN)
__device__ __forceinline__ double raise_to(double m, double a) {
  return bits64(a) > bits64(m) && (unsigned long long)bits64(a) <= 0x7ff0000000000000ull ? a : m;
}
__device__ __forceinline__ float raise_to(float m, float a) { return a > m ? a : m; }
// x + s y for a power of two s: the product is exact, one rounding either way
__device__ __forceinline__ double add_scaled(double x, double s, double y) { return __fma_rn(s, y, x); }
__device__ __forceinline__ float add_scaled(float x, float s, float y) { return __fmaf_rn(s, y, x); }

}  // namespace cgk
