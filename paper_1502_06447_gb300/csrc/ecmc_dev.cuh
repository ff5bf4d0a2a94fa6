// Device/host primitives of the EC library: counter-based random numbers,
// the minimum image, the candidate kinds and the event digest.  The event
// geometry itself (arXiv:1502.06447, Sec. II, Eq. 1) lives in the kernels.
//
// Every FP64 expression is evaluated as written (the library is built with
// -fmad=false; fused multiply-adds only where written as __fma_rn), so the
// event sequence is a pure function of the input state and the Philox key.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define ECMC_HD __host__ __device__ __forceinline__
#else
#define ECMC_HD inline
#endif

namespace ecmc {

// ---------------------------------------------------------------- Philox
// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds of two
// 64x64 -> 128-bit products of the even words with the round multipliers;
// the high halves are xor-ed into the odd words together with the key, the
// words rotate, and the key advances by the two Weyl increments.
struct u64x4 {
  uint64_t v[4];
};

ECMC_HD void mul128(uint64_t a, uint64_t b, uint64_t &hi, uint64_t &lo) {
#ifdef __CUDA_ARCH__
  hi = __umul64hi(a, b);
  lo = a * b;
#else
  unsigned __int128 p = (unsigned __int128)a * b;
  hi = (uint64_t)(p >> 64);
  lo = (uint64_t)p;
#endif
}

ECMC_HD u64x4 philox(uint64_t c0, uint64_t c1, uint64_t c2, uint64_t c3,
                     uint64_t k0, uint64_t k1) {
  const uint64_t m0 = 0xD2E7470EE14C6C93ull, m1 = 0xCA5A826395121157ull;
  const uint64_t w0 = 0x9E3779B97F4A7C15ull, w1 = 0xBB67AE8584CAA73Bull;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    uint64_t h0, l0, h1, l1;
    mul128(m0, c0, h0, l0);
    mul128(m1, c2, h1, l1);
    const uint64_t n0 = h1 ^ c1 ^ k0;
    const uint64_t n2 = h0 ^ c3 ^ k1;
    c0 = n0;
    c1 = l1;
    c2 = n2;
    c3 = l0;
    k0 += w0;
    k1 += w1;
  }
  u64x4 r;
  r.v[0] = c0;
  r.v[1] = c1;
  r.v[2] = c2;
  r.v[3] = c3;
  return r;
}

// random-number layout: key (seed, replica); counter (tag | ec << 8, sweep,
// unit, attempt).  Tags: 1 start bead + direction, 2 tile shift, 3 swap,
// 4 lattice jitter, 5 phantom chains, 6 spring energies (counter word 3 =
// the event index within the EC).
enum : uint64_t {
  TAG_START = 1, TAG_SHIFT = 2, TAG_SWAP = 3, TAG_JITTER = 4, TAG_PHANTOM = 5, TAG_SPRING = 6
};

// top 53 bits -> [0,1)
ECMC_HD double unit53(uint64_t w) { return (double)(w >> 11) * (1.0 / 9007199254740992.0); }

// floor(w * m / 2^64) in [0, m)
ECMC_HD int64_t scale_below(uint64_t w, uint64_t m) {
  uint64_t hi, lo;
  mul128(w, m, hi, lo);
  (void)lo;
  return (int64_t)hi;
}

// ---------------------------------------------------------------- geometry
// Candidate kinds in tie-break order: an exact tie in x goes to the smaller
// kind, then to the smaller partner id.
enum : int { KIND_END = 0, KIND_PASS = 1, KIND_WALL = 2, KIND_HS = 3, KIND_TETHER = 4 };

// ---------------------------------------------------------------- sqrt, quotient
// IEEE double square root and quotient (round to nearest even) in integer
// arithmetic.  GB300 takes 55-60 cycles for a dependent FP64 operation and
// the FP64 pipe 16 cycles of an SM for each FP64 warp instruction, so the
// iterations behind sqrt() and / were the longest links of an event step; a
// dependent 32-bit multiply-add takes about 4.  A lone warp's dependent chain:
// sqrt() 580 cycles, sqrt_rn 280, / 550, div_rn 320.  Both functions take a 22-bit estimate from the FP32 hardware
// approximation, correct it twice by the exact remainder (64-bit wrapping
// arithmetic: the remainders are known to be small), and settle the last
// bit by the sign of one more exact remainder, so the result does not depend
// on the estimate's rounding.
#ifdef __CUDACC__
// An FP64 instruction takes its unit 64 cycles, a comparison or conversion
// more, and the compiler knows several ways to bring back one that the source
// avoids.  Bits of a double go through an empty-handed move, since it turns
// sign tests into FP64 comparisons and a flipped sign bit into a subtraction
// from zero when it sees where they come from.  Operations off the common path
// are calls: it turns a short branch into predicates, and a predicated FP64
// instruction takes its 64 cycles even when no lane wants it.
__device__ __forceinline__ uint64_t bits_of(double x) {
  uint64_t b;
  asm("mov.b64 %0, %1;" : "=l"(b) : "d"(x));
  return b;
}
__device__ __forceinline__ double from_bits(uint64_t b) {
  double x;
  asm("mov.b64 %0, %1;" : "=d"(x) : "l"(b));
  return x;
}
static __device__ __noinline__ double add_fp64(double a, double b) { return a + b; }
static __device__ __noinline__ double square_fp64(double d) { return d * d; }
static __device__ __noinline__ double sqrt_fp64(double a) { return sqrt(a); }
static __device__ __noinline__ double div_fp64(double a, double b) { return a / b; }

// -x
__device__ __forceinline__ double flip(double x) { return from_bits(bits_of(x) ^ 0x8000000000000000ull); }
// |x| with the opposite sign of b's bits
__device__ __forceinline__ double against(double x, uint64_t b) { return from_bits(bits_of(x) ^ (~b & 0x8000000000000000ull)); }

// minimum image of one coordinate difference (|d| < L): d - L above half,
// d + L below -half
__device__ __forceinline__ double wrap_bits(double d, double L, double half, bool on = true) {
  const uint64_t b = bits_of(d);
  if (on && (b & 0x7FFFFFFFFFFFFFFFull) > bits_of(half)) d = add_fp64(d, against(L, b));
  return d;
}
// a < b for doubles >= 0
__device__ __forceinline__ bool less_pos(double a, double b) {
  return bits_of(a) < bits_of(b);
}

// FP32 value of a double, rounded towards zero, by integer operations (the
// conversion instruction takes as long as an FP64 operation); magnitudes
// below 2^-126 give 0, above 2^127 are not used
__device__ __forceinline__ float f32_trunc(double x) {
  const uint64_t b = bits_of(x);
  const unsigned hi = (unsigned)(b >> 32);
  const unsigned f = ((unsigned)(b >> 29) - (384u << 23)) & 0x7FFFFFFFu;
  return __uint_as_float((hi & 0x80000000u) | ((hi & 0x7FFFFFFFu) < (897u << 20) ? 0u : f));
}
// an FP32 value above x >= 0
__device__ __forceinline__ float f32_above(double x) {
  return __uint_as_float(__float_as_uint(f32_trunc(x)) + 1u);
}

// y0 in [1/2, 1) as an integer times 2^-31
__device__ __forceinline__ uint32_t seed_q31(float y) {
  y = fminf(fmaxf(y, 0.5f), 0.99999994f);
  return ((__float_as_uint(y) & 0x7FFFFFu) | 0x800000u) << 7;
}

// a = M 2^E with M in [2^52, 2^54), E even; m = M 2^-52 in [1, 4).
// With y0 = (1 + d) / sqrt(m), |d| < 2^-21.5, s0 = m y0 has remainder
// |m - s0^2| < 2^-18.4; s1 = s0 + (m - s0^2) y0 / 2 errs by less than
// 2^-40.6, its remainder is below 2^-38.6 (exact in units of 2^-90), and
// s2 = s1 + (m - s1^2) y0 / 2 errs by less than 2^-59.  The result is then
// R = floor(s2 2^52) or R + 1: sqrt(M 2^52) > R + 1/2 exactly when
// M 2^52 > R^2 + R (an integer square root is never half-way).
__device__ __forceinline__ double sqrt_rn(double a) {
  const uint64_t b = bits_of(a);
  const unsigned e = (unsigned)(b >> 52);
  if (e - 1u >= 2046u) return sqrt_fp64(a);  // zero, subnormal, negative, inf, nan
  const unsigned even = ~e & 1u;
  const uint64_t M = ((b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << even;
  const float mf = __uint_as_float(((127u + even) << 23) | ((unsigned)(b >> 29) & 0x7FFFFFu));
  const uint32_t y = seed_q31(rsqrtf(mf));                       // Q31
  const uint32_t s0 = __umulhi((uint32_t)(M >> 22), y << 1);     // Q30
  const int64_t r0 = (int64_t)((M << 8) - (uint64_t)s0 * s0);    // Q60, < 2^41.7
  const int64_t s1 = ((int64_t)((uint64_t)s0 << 32)) + (((int64_t)(int32_t)(r0 >> 12) * (int32_t)y) >> 18);  // Q62
  const uint64_t t = (uint64_t)s1 >> 17;                         // Q45
  const int64_t r1 = (int64_t)((M << 38) - t * t);               // Q90, < 2^51.5
  const int64_t s2 = (int64_t)(t << 17) + (((int64_t)(int32_t)(r1 >> 22) * (int32_t)y) >> 38);  // Q62
  const uint64_t R = (uint64_t)s2 >> 10;
  const int64_t d = (int64_t)((M << 52) - R * R - R);
  const uint64_t out = ((uint64_t)((e + 1023u) >> 1) << 52) + (R - 0x0010000000000000ull) + (d > 0 ? 1u : 0u);
  return from_bits(out);
}

// a / b = rho 2^k with rho = Ma / Mb in [1, 2) (Ma doubled when below Mb).
// With y0 = (1 + d) / (Mb 2^-52), |d| < 2^-21.9, q0 = Ma y0 (Q28) errs by
// less than 2^-20.8, q1 = q0 + (rho - q0) by less than 2^-42, q2 by less
// than 2^-59; the last bit follows from the exact remainder (no quotient of
// two doubles is half-way).
__device__ __forceinline__ double div_rn(double a, double b) {
  const uint64_t ab = bits_of(a), bb = bits_of(b);
  const unsigned ea = (unsigned)(ab >> 52) & 0x7FFu, eb = (unsigned)(bb >> 52) & 0x7FFu;
  uint64_t Ma = (ab & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  const uint64_t Mb = (bb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull;
  const unsigned less = Ma < Mb ? 1u : 0u;
  const int eq = (int)ea - (int)eb + 1023 - (int)less;
  if (ea - 1u >= 2046u || eb - 1u >= 2046u || eq < 1 || eq > 2045) return div_fp64(a, b);
  Ma <<= less;
  const float bf = __uint_as_float(0x3F800000u | ((unsigned)(bb >> 29) & 0x7FFFFFu));
  const uint32_t y = seed_q31(__fdividef(1.f, bf));                         // Q31
  const uint32_t q0 = __umulhi((uint32_t)(Ma >> 22), y) >> 1;         // Q30 Q31 / 2^33 = Q28
  const int64_t r0 = (int64_t)((Ma << 28) - (uint64_t)q0 * Mb);       // Q80 of (rho - q0) b, < 2^60.3
  const int64_t q1 = ((int64_t)((uint64_t)q0 << 17)) + (((int64_t)(int32_t)(r0 >> 30) * (int32_t)y) >> 36);  // Q45
  const int64_t r1 = (int64_t)((Ma << 45) - (uint64_t)q1 * Mb);       // Q97, < 2^56
  const int64_t q2 = (q1 << 7) + (((int64_t)(int32_t)(r1 >> 26) * (int32_t)y) >> 50);  // Q52
  const int64_t rem = (int64_t)((Ma << 52) - (uint64_t)q2 * Mb);
  const uint64_t Q = (uint64_t)q2 + (2 * rem > (int64_t)Mb ? 1ull : (2 * rem < -(int64_t)Mb ? ~0ull : 0ull));
  const uint64_t out = (((uint64_t)(unsigned)eq) << 52) + (Q - 0x0010000000000000ull);
  return from_bits(out | ((ab ^ bb) & 0x8000000000000000ull));
}

// d * d, for use where the FP64 units are the limit and the integer units can
// take a share of the work beside them (some 25 instructions).  X = M 2^11 in
// [2^63, 2^64); the upper 64 bits of X^2 are xh^2 + (2 xh xl + ...) >> 32, of
// which h falls short by less than 3.  Half an ulp added, the bits below the
// mantissa tell whether that could matter (three cases in 1024: the FP64
// multiplication decides).
__device__ __forceinline__ double square_rn(double d) {
  const uint64_t b = bits_of(d);
  const unsigned hi = (unsigned)(b >> 32);
  const int e = (int)((hi >> 20) & 0x7FFu);
  const unsigned xh = 0x80000000u | (unsigned)((b << 11) >> 32), xl = (unsigned)b << 11;
  const uint64_t h = (uint64_t)xh * xh + ((uint64_t)__umulhi(xh, xl) << 1);
  const unsigned top = (unsigned)(h >> 63);  // 1: X^2 >= 2^127
  const unsigned sh = 10u + top;
  const uint64_t g = h + (512ull << top);
  const unsigned low = (unsigned)g & ((1024u << top) - 1u);
  // (a carry out of g means the mantissa rounded up to 2^53: left to FP64 too)
  const bool unsure = low - 1u >= (1024u << top) - 3u || g < h || (unsigned)(e - 520) > 999u;
  if (unsure) return square_fp64(d);
  const uint64_t m = g >> sh;  // [2^52, 2^53]: 2^53 carries into the exponent
  const uint64_t out = ((uint64_t)(unsigned)(2 * e - 1023 + (int)top) << 52) + (m - 0x0010000000000000ull);
  return from_bits(out);
}
#endif

// ---------------------------------------------------------------- springs
// Bead-spring chains (Sec. II, ECs with pair potentials): the pieces the EC
// kernels need for a harmonic bond (k/2)(b - sigma)^2.  Host and device
// share them, so the host can check them against other implementations.
#ifdef __CUDA_ARCH__
#define EC_FMA(a, b, c) __fma_rn(a, b, c)
#define EC_SQRT(a) sqrt_rn(a)
#define EC_DIV(a, b) div_rn(a, b)
#else
#define EC_FMA(a, b, c) fma(a, b, c)
#define EC_SQRT(a) sqrt(a)
#define EC_DIV(a, b) ((a) / (b))
#endif

// Natural logarithm of u in (0, 1]: u = m 2^e with m in [sqrt(1/2), sqrt(2)),
// log u = e ln 2 + 2 atanh(z), z = (m - 1)/(m + 1), atanh(z)/z =
// sum_{n=0..14} z^(2n)/(2n + 1) by Horner's rule, ln 2 rounded to double.
// Only +, -, *, / and exact bit moves: every implementation taking these
// steps gets the same bits (within a few ulp of the exact logarithm).
ECMC_HD double ec_log(double u) {
  uint64_t b;
  memcpy(&b, &u, sizeof(b));
  int e = (int)((b >> 52) & 0x7FF) - 1023;
  const uint64_t mb = (b & 0x000FFFFFFFFFFFFFull) | 0x3FF0000000000000ull;
  double m;
  memcpy(&m, &mb, sizeof(m));
  if (mb > 0x3FF6A09E667F3BCDull) {  // m > sqrt(2) rounded to double; both in [1, 2)
    m = m * 0.5;
    e += 1;
  }
  const double z = EC_DIV(m - 1.0, m + 1.0);
  const double z2 = z * z;
  double s = 1.0 / 29.0;
  for (int n = 13; n >= 0; --n) s = s * z2 + 1.0 / (double)(2 * n + 1);
  return (double)e * 0.6931471805599453 + 2.0 * z * s;
}

// Boltzmann energy of one bond at one event from a Philox word:
// dE = -log(u), u = 1 - unit53(w) in (0, 1]
ECMC_HD double spring_dE(uint64_t w) { return -ec_log(1.0 - unit53(w)); }

// Spring event: a pivot at separation d = r_pivot - r_bonded moving along
// unit v may go on until the energy its move adds reaches dE.  Hard spheres
// keep b >= sigma, so the energy falls up to the closest approach along the
// path and rises after it (or from the start when d.v >= 0); dE is spent
// on the rise: b_t = sigma + sqrt((b_s - sigma)^2 + 2 dE / k) with b_s the
// bond length where the rise starts, x = -d.v + sqrt(b_t^2 - |d_perp|^2).
// spring_flight: from dv = d.v, dd = d.d and dEk = 2 dE / k (signs are read
// off the bit patterns: a comparison is an FP64 instruction on the device).
ECMC_HD bool neg_bits(double x) {
  int64_t b;
#ifdef __CUDA_ARCH__
  b = (int64_t)bits_of(x);
#else
  memcpy(&b, &x, sizeof(b));
#endif
  return b < 0 && ((uint64_t)b << 1) != 0;
}
ECMC_HD double spring_flight(double dv, double dd, double sigma, double dEk) {
  double perp2 = EC_FMA(-dv, dv, dd);
  if (neg_bits(perp2)) perp2 = 0.0;
  const double bs = EC_SQRT(neg_bits(dv) ? perp2 : dd);
  const double e = bs - sigma;
  const double bt = sigma + EC_SQRT(e * e + dEk);
  // b_t >= b_s >= |d_perp| exactly; rounding can leave the radicand a few
  // ulp below zero when dE ~ 0 and the path grazes the closest approach
  double rad = bt * bt - perp2;
  if (neg_bits(rad)) rad = 0.0;
  const double x = -dv + EC_SQRT(rad);
  return neg_bits(x) ? 0.0 : x;
}
ECMC_HD double spring_x(double d0, double d1, double d2, double v0, double v1, double v2,
                        double sigma, double k, double dE, double &dv) {
  dv = EC_FMA(d2, v2, EC_FMA(d1, v1, d0 * v0));
  const double dd = EC_FMA(d2, d2, EC_FMA(d1, d1, d0 * d0));
  return spring_flight(dv, dd, sigma, EC_DIV(2.0 * dE, k));
}

ECMC_HD void fnv_mix(uint64_t &h, uint64_t w) {
  h ^= w;
  h *= 0x100000001B3ull;
}

#ifdef __CUDACC__
// FP32 upper bound on a square root from the hardware's fast approximation:
// rsqrtf errs by at most 2 ulp (CUDA's accuracy tables), so after the product
// the relative error is below 4e-7 and the factor 1 + 1e-6 gives a bound.  The
// argument is raised to 1e-30 inside rsqrtf: this keeps 0 finite and moves a
// result by less than 1e-15 in absolute terms, far inside the screen's margin
// eps_v.
__device__ __forceinline__ float sqrt_hi(float y) { return y * rsqrtf(fmaxf(y, 1e-30f)) * 1.000001f; }
#endif

}  // namespace ecmc
