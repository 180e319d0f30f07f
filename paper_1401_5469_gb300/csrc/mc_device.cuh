// Device helpers of the transport kernels: the Philox4x32-10 draw stream,
// integer comparison keys of binary64 values, and the binary64
// logarithm and reciprocal used on the hot path.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "mc_internal.h"

namespace mcgpu {

// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds of two
// 32x32->64-bit products mixed with the other counter words and the key,
// the key advancing by the two Weyl increments between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c.x, hi0 = __umulhi(0xD2511F53u, c.x);
    const uint32_t lo1 = 0xCD9E8D57u * c.z, hi1 = __umulhi(0xCD9E8D57u, c.z);
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// Per-packet uniform stream.  Draw d uses Philox block d/2 with counter
// (d/2, packet, iteration, 0); words (x,y) for even d, (z,w) for odd d;
// u53 = (wa >> 5) 2^26 + (wb >> 6).
struct DrawStream {
  uint32_t k0, k1, packet, iteration;
  uint32_t d, spare_a, spare_b;

  __device__ __forceinline__ void init(uint32_t key0, uint32_t key1, uint32_t pid, uint32_t it) {
    k0 = key0; k1 = key1; packet = pid; iteration = it; d = 0; spare_a = 0; spare_b = 0;
  }
  __device__ __forceinline__ uint64_t next_u53() {
    uint32_t wa, wb;
    if ((d & 1u) == 0u) {
      const uint4 o = philox4x32_10(make_uint4(d >> 1, packet, iteration, 0u), k0, k1);
      wa = o.x; wb = o.y; spare_a = o.z; spare_b = o.w;
    } else {
      wa = spare_a; wb = spare_b;
    }
    ++d;
    return u53_of(wa, wb);
  }
  static __device__ __forceinline__ uint64_t u53_of(uint32_t wa, uint32_t wb) {
    return (static_cast<uint64_t>(wa >> 5) << 26) | static_cast<uint64_t>(wb >> 6);
  }
  // z in (0, 1]
  __device__ __forceinline__ double open0() { return __ull2double_rn(next_u53() + 1ull) * 0x1.0p-53; }
  // z in [0, 1)
  __device__ __forceinline__ double closed0() { return __ull2double_rn(next_u53()) * 0x1.0p-53; }
  // mu = 2 z - 1 for z = u53 2^-53 in [0, 1): (u53 - 2^52) 2^-52, exact.
  // Assembled from the integer's bits (no conversion instruction).
  static __device__ __forceinline__ double mu_from_u53(unsigned long long u) {
    const long long v = static_cast<long long>(u) - (1ll << 52);
    const unsigned long long a = static_cast<unsigned long long>(v < 0 ? -v : v);  // <= 2^52
    if (a == 0ull) return 0.0;
    const int lz = __clzll(static_cast<long long>(a));
    const unsigned long long mant = ((a << lz) << 1) >> 12;
    const unsigned long long bits = (static_cast<unsigned long long>(63 - lz - 52 + 1023) << 52) |
                                    mant | (v < 0 ? (1ull << 63) : 0ull);
    return __longlong_as_double(static_cast<long long>(bits));
  }
};

// The bit pattern of a binary64 value read as a signed integer.  Compared
// with the pattern of a positive value (or +0) it orders exactly like the
// values do, negative values included (their patterns are negative
// integers), so every comparison in the transport kernels -- each has one
// operand known to be positive -- runs on the integer pipe.
__device__ __forceinline__ long long rawkey(double v) { return __double_as_longlong(v); }

// Pattern of -inf: below every non-negative value's pattern.
constexpr long long kKeyNegInf = (long long)0xfff0000000000000ll;

// A pattern below that of every non-negative value.
constexpr long long kRawBelowZero = (long long)0x8000000000000000ll;

// binary64 -> binary32 toward zero on the bit pattern, any sign: |result| <=
// |d| with a relative error below 2^-23, values below the binary32 normal
// range give (signed) 0, values above its range (and NaN) +-infinity.
__device__ __forceinline__ float f32_rz_any(double d) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(d));
  const int e = static_cast<int>((b >> 52) & 0x7ffull) - 1023 + 127;
  const unsigned int mag = e <= 0 ? 0u
                           : e >= 255 ? 0x7f800000u
                                      : (static_cast<unsigned int>(e) << 23) |
                                            static_cast<unsigned int>((b >> 29) & 0x7fffffull);
  return __int_as_float(static_cast<int>(mag | (static_cast<unsigned int>(b >> 63) << 31)));
}

// The same for |d| < 2^127 (fewer instructions): below the binary32 normal
// range (signed) 0.
__device__ __forceinline__ float f32_rz_small(double d) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(d)), lo = static_cast<uint32_t>(__double2loint(d));
  const uint32_t a = hi & 0x7fffffffu;
  const uint32_t m = __funnelshift_l(lo, a - 0x38000000u, 3);  // the exponent rebiased, 23 fraction bits
  return __uint_as_float((a >= 0x38100000u ? m : 0u) | (hi & 0x80000000u));
}

// The same for a depth: at most the largest finite value.
__device__ __forceinline__ float f32_rz_below_inf(double d) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(d)), lo = static_cast<uint32_t>(__double2loint(d));
  const uint32_t a = min(hi & 0x7fffffffu, 0x47efffffu);
  const uint32_t m = __funnelshift_l(lo, a - 0x38000000u, 3);
  return __uint_as_float((a >= 0x38100000u ? m : 0u) | (hi & 0x80000000u));
}

// v < 0, excluding -0 (its pattern is the most negative integer).
__device__ __forceinline__ bool strictly_negative(double v) {
  const long long b = __double_as_longlong(v);
  return b < 0 && b != kRawBelowZero;
}

// A 32-bit word the host may write while the kernel runs (pinned, mapped
// host memory): system-scope load, so the host's store becomes visible.
__device__ __forceinline__ uint32_t load_sys_u32(const uint32_t *a) {
  uint32_t v;
  asm volatile("ld.relaxed.sys.global.u32 %0, [%1];" : "=r"(v) : "l"(a) : "memory");
  return v;
}

// L2 eviction priority for the J_blue sums: a J_blue array is as large as the
// Sobolev depths (S x L cells) and is only written, by atomics, during a
// transport launch; marking those atomics evict-first keeps the line list,
// the depths and the branching records -- what the random walks read on
// their dependency chains -- resident in L2 instead.
__device__ __forceinline__ unsigned long long l2_evict_first_policy() {
  unsigned long long pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void red_add_evict_first(double *a, double v, unsigned long long pol) {
  asm volatile("red.global.add.L2::cache_hint.f64 [%0], %1, %2;" ::"l"(a), "d"(v), "l"(pol) : "memory");
}
__device__ __forceinline__ void red_add_evict_first(unsigned long long *a, unsigned long long v,
                                                    unsigned long long pol) {
  asm volatile("red.global.add.L2::cache_hint.u64 [%0], %1, %2;" ::"l"(a), "l"(v), "l"(pol) : "memory");
}

// Read-only loads that are issued where they stand: the compiler may move a
// plain load down to its first use, and on a lone walk the instructions
// between the two are what its latency hides behind.
__device__ __forceinline__ unsigned long long load_here(const void *a) {
  unsigned long long v;
  asm volatile("ld.global.nc.b64 %0, [%1];" : "=l"(v) : "l"(a));
  return v;
}
__device__ __forceinline__ uint32_t load_here32(const void *a) {
  uint32_t v;
  asm volatile("ld.global.nc.b32 %0, [%1];" : "=r"(v) : "l"(a));
  return v;
}
__device__ __forceinline__ float load_here_f(const float *a) {
  float v;
  asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(v) : "l"(a));
  return v;
}
__device__ __forceinline__ uint4 load_here4(const void *a) {
  uint4 v;
  asm volatile("ld.global.nc.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(a));
  return v;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Reciprocal and square root on the integer pipe.  A binary64 instruction
// occupies its sub-partition's pipe for 64 cycles, and its result reaches another
// pipe 45 cycles later than the next binary64 instruction; a 32 x 32 -> 64-bit
// product takes 4.  Both start from the binary32 approximation of the 53-bit
// significand (24 bits), and take two corrections: the residual exactly, as a
// 64-bit integer (its upper bits cancel, so that products modulo 2^64 are
// enough), the correction residual / slope in binary32 with the same
// approximation.  The first leaves 2^-42 (its rounding and the omitted second-order
// term); the second is taken downward, so that the sum is the exact value cut to 1/32
// (reciprocal) or 1/16 ulp and rounding it to 53 bits rounds the value: within 0.501
// ulp and without a bias (tested on the device over every binary32 prefix of the
// significand through mc_selftest_math).  Rounded to nearest instead, the second left
// half of such a unit in the mean, which a packet's 1/nu collects: frequencies of walks
// of up to 2e4 electron scatterings were 2.0e-10 off (rms), now 3.2e-11.  Newton's iteration in residual form (J.-M. Muller,
// Elementary Functions, ch. 2).  Before: three and five binary64 instructions
// from rcp.approx / rsqrt.approx.f64, within 1 ulp.

// round(a b) for |a b| < 2^21, through the low bits of a binary32 sum.
__device__ __forceinline__ int32_t mul_round(float a, float b) {
  return __float_as_int(fmaf(a, b, 12582912.0f)) - 0x4b400000;
}

// floor(a b), likewise.
__device__ __forceinline__ int32_t mul_floor(float a, float b) {
  return __float_as_int(__fmaf_rd(a, b, 12582912.0f)) - 0x4b400000;
}

// 1/x for normal |x| in [2^-1000, 2^1000].  HERE: evaluated only where it
// stands (the compiler may otherwise evaluate it ahead of the branch that needs it).
template <bool HERE = false>
__device__ __forceinline__ double rcp64(double x) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const uint32_t e = (hi >> 20) & 0x7ffu;
  const uint32_t mh = (hi & 0xfffffu) | 0x100000u;  // the significand's upper 21 bits
  const unsigned long long m = (static_cast<unsigned long long>(mh) << 32) | lo;  // 2^52 times [1, 2)
  const float f32 = static_cast<float>(__funnelshift_l(lo, mh, 11));
  float y;  // 2^-31 / significand
  if (HERE) asm volatile("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f32));
  else asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f32));
  const float t = fminf(fmaxf(y * 0x1.0p55f, 0x1.0p23f), 0x1.fffffep23f);
  const uint32_t q0 = (__float_as_uint(t) & 0x7fffffu) | 0x800000u;  // units of 2^-24
  const long long r0 = static_cast<long long>(0ull - m * q0);        // 2^76 - m q0
  const int32_t c1 = mul_round(static_cast<float>(static_cast<int32_t>(r0 >> 24)), y * 0x1.0p22f);
  const unsigned long long q1 = (static_cast<unsigned long long>(q0) << 19) +
                                static_cast<unsigned long long>(static_cast<long long>(c1));  // 2^-43
  const long long r1 = static_cast<long long>(0ull - m * q1);        // 2^95 - m q1
  const int32_t c2 = mul_floor(static_cast<float>(static_cast<int32_t>(r1 >> 26)), y * 0x1.0p20f);
  const unsigned long long f = (q1 << 15) + static_cast<unsigned long long>(static_cast<long long>(c2));  // 2^-58
  const unsigned long long bits = (static_cast<unsigned long long>(2044u - e) << 52) + ((f + 16ull) >> 5);
  return __longlong_as_double(static_cast<long long>(bits | (static_cast<unsigned long long>(hi & 0x80000000u) << 32)));
}

// Square root of a normal x > 0; sqrt64: of 0 too.
__device__ __forceinline__ double sqrt64_pos(double x) {
  const uint32_t hi = static_cast<uint32_t>(__double2hiint(x)), lo = static_cast<uint32_t>(__double2loint(x));
  const uint32_t e = hi >> 20, odd = ~e & 1u;
  const unsigned long long m = (static_cast<unsigned long long>((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const unsigned long long a = m << (10u + odd);  // 2^62 times [1, 4)
  const float f = static_cast<float>(static_cast<uint32_t>(a >> 32));
  float y;  // 2^-15 / sqrt
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
  const float t = fminf(fmaxf(f * y, 0x1.0p15f), 0x1.fffffep15f);
  const uint32_t s0 = ((__float_as_uint(t) & 0x7fffffu) | 0x800000u) << 8;  // units of 2^-31
  const long long r0 = static_cast<long long>(a - static_cast<unsigned long long>(s0) * s0);
  const int32_t c1 = mul_round(static_cast<float>(static_cast<int32_t>(r0 >> 13)), y * 0x1.0p7f);
  const unsigned long long s1 = (static_cast<unsigned long long>(s0) << 11) +
                                static_cast<unsigned long long>(static_cast<long long>(c1));  // 2^-42
  const long long r1 = static_cast<long long>((a << 22) - s1 * s1);
  const int32_t c2 = mul_floor(static_cast<float>(static_cast<int32_t>(r1 >> 14)), y);
  const unsigned long long s2 = (s1 << 14) + static_cast<unsigned long long>(static_cast<long long>(c2));  // 2^-56
  const unsigned long long bits =
      (static_cast<unsigned long long>(((e + 1023u - odd) >> 1) - 1u) << 52) + ((s2 + 8ull) >> 4);
  return __longlong_as_double(static_cast<long long>(bits));
}
__device__ __forceinline__ double sqrt64(double x) {
  return __double_as_longlong(x) == 0ll ? 0.0 : sqrt64_pos(x);
}

// ln(2) split so that k * kLn2Head is exact for |k| < 2^20.
constexpr double kLn2Head = 0x1.62e42fee00000p-1;
constexpr double kLn2Tail = 0x1.a39ef35793c76p-33;

// {c = 1/F, -ln(c)} per breakpoint F; see gen_log_table.py.
static __constant__ double2 c_log_tab[128] = {
#include "mc_log_table.inc"
};

// ln(m 2^k) for m in [1, 2) given by its 52 fraction bits, by Tang's
// table-driven method (ACM TOMS 16, 1990): m is moved to [0.75, 1.5) (k
// adjusted), r = m c - 1 with the nearest breakpoint's c = 1/F, and
// ln(1 + r) from its Taylor series to degree 8 (|r| < 2^-7).
__device__ __forceinline__ double log_core(int k, unsigned long long frac) {
  const int i = static_cast<int>(frac >> 45);
  long long mb = static_cast<long long>(0x3ff0000000000000ull | frac);
  if (i >= 64) { mb -= (1ll << 52); ++k; }  // m / 2, exponent field only
  const double m = __longlong_as_double(mb);
  const double2 ct = c_log_tab[i];
  const double r = fma(m, ct.x, -1.0);
  double p = -0.125;
  p = fma(p, r, 1.0 / 7.0);
  p = fma(p, r, -1.0 / 6.0);
  p = fma(p, r, 0.2);
  p = fma(p, r, -0.25);
  p = fma(p, r, 1.0 / 3.0);
  p = fma(p, r, -0.5);
  p = fma(p, r, 1.0);
  const double dk = static_cast<double>(k);
  return fma(dk, kLn2Head, ct.y) + fma(p, r, dk * kLn2Tail);
}

#define MC_KLN2(k) {(k) * kLn2Head, (k) * kLn2Tail}
#define MC_KLN2_8(b) MC_KLN2(b), MC_KLN2(b - 1), MC_KLN2(b - 2), MC_KLN2(b - 3), \
                     MC_KLN2(b - 4), MC_KLN2(b - 5), MC_KLN2(b - 6), MC_KLN2(b - 7)
// {k ln2 head, k ln2 tail} for k = 0, -1, ..., -55 (both products exact / correctly rounded).
static __constant__ double2 c_kln2[56] = {MC_KLN2_8(0), MC_KLN2_8(-8), MC_KLN2_8(-16), MC_KLN2_8(-24),
                                          MC_KLN2_8(-32), MC_KLN2_8(-40), MC_KLN2_8(-48)};
#undef MC_KLN2_8
#undef MC_KLN2

// -ln(z) for z = u 2^-53, 1 <= u <= 2^53 (the (0,1] draw): integer-only
// reduction, k ln2 from a table (no conversion instruction), then Tang's
// method as in log_core.
__device__ __forceinline__ double neg_log_u53(unsigned long long u) {
  const int lz = __clzll(static_cast<long long>(u));
  const unsigned long long frac = ((u << lz) << 1) >> 12;
  int k = 63 - lz - 53;  // in [-53, 0]
  const int i = static_cast<int>(frac >> 45);
  long long mb = static_cast<long long>(0x3ff0000000000000ull | frac);
  if (i >= 64) { mb -= (1ll << 52); ++k; }
  const double m = __longlong_as_double(mb);
  const double2 ct = c_log_tab[i];
  const double2 kl = c_kln2[-k];
  const double r = fma(m, ct.x, -1.0);
  double p = -0.125;
  p = fma(p, r, 1.0 / 7.0);
  p = fma(p, r, -1.0 / 6.0);
  p = fma(p, r, 0.2);
  p = fma(p, r, -0.25);
  p = fma(p, r, 1.0 / 3.0);
  p = fma(p, r, -0.5);
  p = fma(p, r, 1.0);
  return -((kl.x + ct.y) + fma(p, r, kl.y));
}

// -ln z in binary32 for the draw z = u 2^-53, 1 <= u <= 2^53, to a relative
// error below 2^-21: z = m 2^e with m in [0.75, 1.5), f = m - 1 from the
// integer (exact to 2^-23 however near 1 the draw is), ln m = 2 atanh(s) with
// s = f / (2 + f), |s| <= 1/5, by its series to s^9 (Abramowitz & Stegun
// 4.1.27; the first omitted term is below 2^-27 of the sum).
__device__ __forceinline__ float neg_log_u53_f(unsigned long long u) {
  const int lz = __clzll(static_cast<long long>(u));
  const unsigned long long m = u << lz;  // [2^63, 2^64)
  const bool up = m >= 0xc000000000000000ull;
  const unsigned long long a = up ? 0ull - m : m - 0x8000000000000000ull;  // |f| 2^64 or 2^63
  const float mag = fmaf(static_cast<float>(static_cast<uint32_t>(a >> 32)), 0x1.0p32f,
                         static_cast<float>(static_cast<uint32_t>(a)));
  const float f = up ? mag * -0x1.0p-64f : mag * 0x1.0p-63f;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(2.0f + f));
  const float s = f * r, s2 = s * s;
  float q = fmaf(s2, 1.0f / 9.0f, 1.0f / 7.0f);
  q = fmaf(s2, q, 0.2f);
  q = fmaf(s2, q, 1.0f / 3.0f);
  const float lnm = 2.0f * fmaf(s * s2, q, s);
  return fmaf(static_cast<float>(lz - 10 - (up ? 1 : 0)), 0x1.62e43p-1f, -lnm);
}

// Downbranch emission (Sect. 2.5): the first entry k of the activated upper
// level's branching row with z < cdf[k], z = u 2^-53.  z < cdf[k] <=> u <
// ceil(cdf[k] 2^53) = thr[k] exactly; the search starts at the guide entry of
// bucket floor(z n), whose slot settles most draws.
// The bucket slot of draw u in the row of rinfo (begin | length << 32):
// floor(u n / 2^53) in two 32-bit products.
__device__ __forceinline__ uint32_t bucket_index(unsigned long long rinfo, unsigned long long u) {
  const uint32_t b = static_cast<uint32_t>(rinfo), len = static_cast<uint32_t>(rinfo >> 32);
  const unsigned long long lo = static_cast<unsigned long long>(static_cast<uint32_t>(u)) * len;
  const unsigned long long s = static_cast<unsigned long long>(static_cast<uint32_t>(u >> 32)) * len + (lo >> 32);
  return b + static_cast<uint32_t>(s >> 21);  // (row offsets are 32-bit: so is every index)
}

__device__ __forceinline__ const DbrSlot *bucket_slot(const DbrSlot *slots, unsigned long long rinfo,
                                                      unsigned long long u) {
  return slots + bucket_index(rinfo, u);
}

__device__ __forceinline__ void load_slot(const DbrSlot *slot, uint4 &a, uint4 &c) {
  a = __ldg(reinterpret_cast<const uint4 *>(slot));
  c = __ldg(reinterpret_cast<const uint4 *>(slot) + 1);
}

__device__ __forceinline__ void load_slot_here(const DbrSlot *slot, uint4 &a, uint4 &c) {
  a = load_here4(slot);
  c = load_here4(reinterpret_cast<const uint4 *>(slot) + 1);
}

// The same in four 64-bit loads: the mixed kernel's lone walk took 91 ms with
// them instead of 102 (the binary64 kernel's 105 instead of 100).
__device__ __forceinline__ void load_slot_here64(const DbrSlot *slot, uint4 &a, uint4 &c) {
  const unsigned long long *w = reinterpret_cast<const unsigned long long *>(slot);
  const unsigned long long w0 = load_here(w), w1 = load_here(w + 1), w2 = load_here(w + 2), w3 = load_here(w + 3);
  a = make_uint4(static_cast<uint32_t>(w0), static_cast<uint32_t>(w0 >> 32), static_cast<uint32_t>(w1),
                 static_cast<uint32_t>(w1 >> 32));
  c = make_uint4(static_cast<uint32_t>(w2), static_cast<uint32_t>(w2 >> 32), static_cast<uint32_t>(w3),
                 static_cast<uint32_t>(w3 >> 32));
}

// The emitted line from a loaded slot {thr[3], emit[0]}, {emit[1], emit[2],
// guide, -}, or -1: u's upper 32 bits equal a threshold's, or u lies behind
// the slot's entries.
__device__ __forceinline__ int32_t slot_line(uint4 a, uint4 c, unsigned long long u) {
  const uint32_t v = static_cast<uint32_t>(u >> 21);
  uint32_t line = a.w;
  if (v >= a.x) line = (v > a.x && v < a.y) ? c.x : (v > a.y && v < a.z) ? c.y : 0xffffffffu;
  return static_cast<int32_t>(line);
}

// The row's entries one by one from position i (the last has thr = 2^53 > u).
__device__ __forceinline__ int32_t search_row(const DbrRec *rec, uint32_t i, unsigned long long u) {
  while (u >= __ldg(&rec[i].thr)) ++i;
  return static_cast<int32_t>(__ldg(&rec[i].emit));
}

// Lone walk (all 32 lanes converged): 32 entries of the row per coalesced load
// (lane i takes entry i), the first with u below its threshold by a vote.
__device__ __forceinline__ int32_t search_row_lone(const DbrRec *rec, unsigned long long rinfo, uint32_t guide,
                                                   unsigned long long u, unsigned lane) {
  const uint32_t end = static_cast<uint32_t>(rinfo) + static_cast<uint32_t>(rinfo >> 32);
  for (uint32_t i0 = static_cast<uint32_t>(rinfo) + guide;; i0 += 32u) {
    const uint32_t i = i0 + lane;
    ulonglong2 r = make_ulonglong2(~0ull, 0ull);  // lanes past the row's end vote yes
    if (i < end) r = __ldg(reinterpret_cast<const ulonglong2 *>(rec + i));
    const unsigned m = __ballot_sync(0xffffffffu, u < r.x);
    if (m != 0u)
      return __shfl_sync(0xffffffffu, static_cast<int32_t>(static_cast<uint32_t>(r.y)), __ffs(m) - 1);
  }
}

// Constants of a segment's line scan in binary32 (the error budget stands at
// the binary64 kernel's scan).
struct ScanF {
  unsigned long long mc;  // significand of nu_cmf
  int ec;                 // its exponent field
  float lf, tf;           // path length per unit of significand difference; kappa' D
  float tau;              // the optical-depth draw
  float lx, mx;           // path length to the shell exit and its error bound (infinite: not known)
};

// The frequency's part of it; Df = D in binary32.
__device__ __forceinline__ void scan_frequency(ScanF &f, double nu_cmf, float Df) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(nu_cmf));
  f.ec = static_cast<int>(b >> 52);
  f.mc = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  float im;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(im) : "f"(static_cast<float>(static_cast<uint32_t>(f.mc >> 29))));
  f.lf = (Df * im) * 0x1.0p-29f;
}

// Significand difference nu_cmf - nu_line in units of nu_cmf's last place, as
// binary32 (0 when the line is not below nu_cmf); ok: the line's binade is
// nu_cmf's or a lower one.
__device__ __forceinline__ float scan_delta(const ScanF &f, long long line_bits, bool &ok) {
  const unsigned long long b = static_cast<unsigned long long>(line_bits);
  const int sh = f.ec - static_cast<int>(b >> 52);
  ok = sh >= 0;
  const unsigned long long m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  const long long d = static_cast<long long>(f.mc) - static_cast<long long>(m >> (sh < 63 ? sh & 63 : 63));
  const float v = fmaf(static_cast<float>(static_cast<uint32_t>(d >> 32)), 0x1.0p32f,
                       static_cast<float>(static_cast<uint32_t>(d)));
  return d > 0 ? v : 0.0f;
}

// Draws of a lone walk in the mixed kernel, computed ahead by the whole warp:
// a draw's value depends only on (key, packet, iteration, draw index), so lane i
// computes Philox block base/2 + i and the walk reads its next 64 draws from
// shared memory instead of running Philox on its own dependency chain.  Values
// are identical to DrawStream's.  All state is warp-uniform.
constexpr uint32_t kWarpDraws = 64;
constexpr uint32_t kNoPacket = 0xffffffffu;

// Draw i of a packet's stream computed on its own, for draws past the end of
// the warp buffer (only a macro atom's long walks get there).  Out of line
// and by value, so that the common path does not evaluate it.
static __device__ __noinline__ unsigned long long u53_past_buffer(uint32_t k0, uint32_t k1, uint32_t packet,
                                                           uint32_t iteration, uint32_t i) {
  const uint4 o = philox4x32_10(make_uint4(i >> 1, packet, iteration, 0u), k0, k1);
  return (i & 1u) ? DrawStream::u53_of(o.z, o.w) : DrawStream::u53_of(o.x, o.y);
}

struct WarpDraws {
  unsigned long long *u;  // [64] u53 of draws base .. base + 63 (shared memory, per warp)
  uint32_t base, pid;     // first draw index held, packet (kNoPacket: none)

  __device__ __forceinline__ void init(unsigned long long *warp_buf) {
    u = warp_buf;
    base = 0u;
    pid = kNoPacket;
  }
  // All 32 lanes hold the walk's draw stream: refill when fewer than the three
  // draws a segment may take are left.
  __device__ __forceinline__ void keep_u(const DrawStream &ds, uint32_t k0, uint32_t k1, uint32_t iteration,
                                         unsigned lane) {
    if (ds.packet == pid && ds.d + 3u <= base + kWarpDraws) return;
    const uint32_t b = ds.d & ~1u;
    const uint4 o = philox4x32_10(make_uint4((b >> 1) + lane, ds.packet, iteration, 0u), k0, k1);
    __syncwarp();  // every lane has read the old contents
    u[2 * lane] = DrawStream::u53_of(o.x, o.y);
    u[2 * lane + 1] = DrawStream::u53_of(o.z, o.w);
    __syncwarp();
    base = b;
    pid = ds.packet;
  }
  // The walk's next draw, from the buffer that keep_u() holds filled.
  __device__ __forceinline__ unsigned long long take_u53(DrawStream &ds) const { return u[ds.d++ - base]; }
  // The draw take_u53 returns next, without taking it.
  __device__ __forceinline__ unsigned long long peek_u53(const DrawStream &ds) const { return u[ds.d - base]; }
};

// A macro atom's internal jumps (Sect. 2.5) by a whole warp (a lone walk): a jump's targets in coalesced
// loads, 32 entries a round, the first with the draw below its threshold by a vote.
template <class Draws>
__device__ __forceinline__ unsigned long long macroatom_walk_lone(const MaRow *rows, const MaJump *jumps, int32_t row,
                                                                  const Draws &md, unsigned lane) {
  for (uint32_t n = 0; n < kMaMaxJumps; ++n) {
    const MaRow *mr = rows + row;
    const unsigned long long thr = __ldg(&mr->jump_thr);
    const uint2 jb = __ldg(reinterpret_cast<const uint2 *>(&mr->jump_begin));  // begin, length
    const uint2 db = __ldg(reinterpret_cast<const uint2 *>(&mr->dbr_begin));
    const unsigned long long za = md.next();
    if (!(za < thr)) return static_cast<unsigned long long>(db.x) | (static_cast<unsigned long long>(db.y) << 32);
    const unsigned long long zb = md.next();
    const MaJump *jp = jumps + jb.x;
    for (uint32_t i0 = 0;; i0 += 32u) {  // (the last threshold is 2^53 > zb; past the end the last entry)
      const uint32_t i = min(i0 + lane, jb.y - 1u);
      const unsigned m = __ballot_sync(0xffffffffu, zb < __ldg(&jp[i].thr));
      const int32_t t = __ldg(&jp[i].target);
      if (m != 0u || i0 + 32u >= jb.y) {
        row = __shfl_sync(0xffffffffu, t, m != 0u ? __ffs(m) - 1 : 31);
        break;
      }
    }
  }
  const uint2 db = __ldg(reinterpret_cast<const uint2 *>(&rows[row].dbr_begin));
  return static_cast<unsigned long long>(db.x) | (static_cast<unsigned long long>(db.y) << 32);
}

// The pool of walks handed over.  A walk is written, then its place marked; a
// taker reads the mark, then claims the place.  Nothing waits: a place given
// out but not yet marked ends a taker's search, and the warp that is filling it
// comes back to the pool after its own walk, so every walk is taken.
__device__ __forceinline__ void pool_put(const TransportParams &p, unsigned place, const PoolWalk &w) {
  p.pool[place] = w;
  __threadfence();
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p.pool_ready + place), "r"(1u) : "memory");
}
// The place of a walk to run, or -1.
__device__ __forceinline__ int pool_take(const TransportParams &p) {
  for (int tries = 0; tries < 256; ++tries) {  // (a failed claim: another warp took that one)
    unsigned long long t, h;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(t) : "l"(p.pool_ctl + 1) : "memory");
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(h) : "l"(p.pool_ctl) : "memory");
    if (t >= h || t >= p.pool_cap) return -1;
    uint32_t ready;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(ready) : "l"(p.pool_ready + t) : "memory");
    if (!ready) return -1;
    if (atomicCAS(p.pool_ctl + 1, t, t + 1ull) == t) return static_cast<int>(t);
  }
  return -1;
}

// First index j with nu[j] < v (nu strictly descending), by a whole warp: 32
// probes a round.
__device__ __forceinline__ int32_t first_redward_warp(const double *nu, int32_t L, double v, unsigned lane) {
  int32_t lo = 0, n = L;  // the answer is in [lo, lo + n]
  while (n > 0) {
    const int32_t step = (n + 31) >> 5;
    const int32_t end = min((static_cast<int32_t>(lane) + 1) * step, n);  // this lane's probe is the last before it
    const unsigned m = __ballot_sync(0xffffffffu, __double_as_longlong(__ldg(nu + lo + end - 1)) <
                                                      __double_as_longlong(v));
    if (m == 0u) return lo + n;
    const int32_t k = __ffs(m) - 1;
    const int32_t to = min((k + 1) * step, n) - 1;  // the answer is at most lo + to
    lo += k * step;
    n = to - k * step;
  }
  return lo;
}

// ln(x) for a positive normal binary64 x.
__device__ __forceinline__ double log_pos(double x) {
  const unsigned long long b = static_cast<unsigned long long>(__double_as_longlong(x));
  return log_core(static_cast<int>((b >> 52) & 0x7ffull) - 1023, b & 0x000fffffffffffffull);
}

}  // namespace mcgpu
