// sv_digits.cuh -- FP64 values as small integers for the FP16 tensor cores (the
// exact contractions of sv_vanka_tc64.cu and sv_apply_tc64.cu).
//
// A strip of 128 cell columns (132 held) is walked two cell rows at a time.  The cells
// in reach of a step share an exponent E: x = 2^(E - 58) q, |x| < 2^E, q an integer
// written in ND = 6 balanced digits of 10 bits (the sweep), or 2^(E - 71) q in 6 digits of
// 12 bits (the operator, whose coefficients leave more of FP32's 24 bits to them).  In shared memory a digit of a cell row
// is a plane of 16 bytes per cell (the FP16 digits of its eight velocity values: Q2
// nodes (2i + PI, 2j + PJ) of component c at 4 c + 2 PJ + PI), so the operand of the
// cells shifted by (dx, dy) is the same memory at another start address.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace sv {
namespace dig {

constexpr int COLS = 128, WCOLS = COLS + 4;      // owned and held cell columns
constexpr int ND = 6;                            // digits of a value
constexpr int PLANE = WCOLS * 16;                // one digit of one cell row
constexpr int ROWB = ND * PLANE;                 // a cell row
// Warp roles.  Accumulators to results: two groups of eight warps (cell row, lane
// quarter) that take the steps in turn, so that one group's arithmetic runs while the
// other reads the next step's accumulators; values to digits: nine warps.
constexpr int EPI_WARPS = 16, EPI_GROUP = 8, SLICE_WARPS = 9;
constexpr int SLICE_T = 32 * SLICE_WARPS;
static_assert(2 * WCOLS <= SLICE_T, "one thread per cell of a row pair");
constexpr int EB_MIN = 200;                      // smallest exponent in use (E + 1022): scales stay normal

// E + 1022 for values below 2^(m - 1022), one binade above them, and whether one in use
// still serves them: a walk then renews it seldom.  0x7ff where a value is not finite.
__device__ __forceinline__ int exp_for(int m) { return m >= 0x7ff ? 0x7ff : max(min(m + 1, 0x7fe), EB_MIN); }
__device__ __forceinline__ bool exp_fits(int m, int eb) { return m <= eb && (eb - m <= 3 || eb == EB_MIN) && (m < 0x7ff) == (eb < 0x7ff); }

// q = x 2^(58 - E) rounded to nearest, |x| < 2^E, eb = E + 1022.  Exact for |x| >=
// 2^(E - 6): the mantissa's 53 bits then lie above the last place.
__device__ __forceinline__ long long to_fixed(double x, int eb) {
  const unsigned hi = __double2hiint(x), lo = __double2loint(x);
  const int e = (hi >> 20) & 0x7ff, d = eb - e;
  const unsigned long long m = (static_cast<unsigned long long>((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  // zero and subnormals: d >= EB_MIN shifts everything out
  const unsigned long long v = (((m << 6) >> min(d, 63)) + 1) >> 1;
  return static_cast<int>(hi) < 0 ? -static_cast<long long>(v) : static_cast<long long>(v);
}

constexpr unsigned long long digit_bias() {
  unsigned long long b = 0;
  for (int k = 0; k < ND; ++k) b |= 512ull << (10 * k);
  return b;
}

// digit j (0 the highest) of two biased words as FP16 integers in [-512, 511]
__device__ __forceinline__ unsigned digit2(unsigned long long a, unsigned long long b, int j) {
  const int s = 10 * (ND - 1 - j);
  const unsigned t = (static_cast<unsigned>(a >> s) & 0x3ffu) | ((static_cast<unsigned>(b >> s) & 0x3ffu) << 16) | 0x64006400u;
  __half2 h;
  memcpy(&h, &t, 4);
  h = __hadd2(h, __half2half2(__ushort_as_half(0xE600)));   // -1536
  unsigned u;
  memcpy(&u, &h, 4);
  return u;
}

// The wide form: six digits of 12 bits in [-2048, 2048], q = x 2^(71 - E) truncated,
// |x| < 2^E.  Nothing is lost of |x| >= 2^(E - 19).  Digits of |q| plus 2048 each: lo the
// four lower ones, hi the upper two.
struct Wide {
  unsigned long long lo;
  unsigned hi;
  float sign;
};
// shifts whose counts of 64 and more (negative ones too) give 0
__device__ __forceinline__ unsigned long long shl64(unsigned long long v, int k) {
  unsigned long long r;
  asm("shl.b64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(k));
  return r;
}
__device__ __forceinline__ unsigned long long shr64(unsigned long long v, int k) {
  unsigned long long r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(k));
  return r;
}
__device__ __forceinline__ Wide to_wide(double x, int eb) {
  constexpr unsigned long long mask = (1ull << 48) - 1, bias = 0x800800800800ull;
  const unsigned h = __double2hiint(x), l = __double2loint(x);
  const int d = eb - static_cast<int>((h >> 20) & 0x7ffu);   // the mantissa's last place: 2^(18 - d) units
  // zero and subnormals: d >= EB_MIN shifts everything out
  const unsigned long long m = (static_cast<unsigned long long>((h & 0xfffffu) | 0x100000u) << 32) | l;
  const unsigned long long b = ((shl64(m, 18 - d) | shr64(m, d - 18)) & mask) + bias;
  Wide w;
  w.lo = b;
  w.hi = static_cast<unsigned>(shr64(m, 30 + d)) + static_cast<unsigned>(b >> 48) + ((2048u << 12) + 2048u);
  w.sign = __uint_as_float((h & 0x80000000u) | 0x3f800000u);
  return w;
}
// digit j (0 the highest) of two values as FP16 integers, exact: 2^23 + 2048 + digit as
// the mantissa of an FP32 number
__device__ __forceinline__ unsigned wide_digit2(const Wide& a, const Wide& b, int j) {
  auto digit = [j](const Wide& w) {
    const unsigned t = j == 0 ? w.hi >> 12 : j == 1 ? w.hi & 0xfffu : static_cast<unsigned>(w.lo >> (12 * (5 - j))) & 0xfffu;
    return fmaf(__uint_as_float(t | 0x4b000000u), w.sign, -8390656.0f * w.sign);
  };
  const __half2 h = __floats2half2_rn(digit(a), digit(b));
  unsigned u;
  memcpy(&u, &h, 4);
  return u;
}

// T += 2^K times a digit sum (an integer in FP32; below 2^(63 - K)), rounded to an integer
// for K < 0
template <int K>
__device__ __forceinline__ void add_digit(long long& t, uint32_t f) {
  static_assert(K <= 48, "weight of a digit sum");
  const float v = __uint_as_float(f);
  if constexpr (K < 0) {
    t += static_cast<long long>(__float2int_rn(v * (1.0f / (1 << -K))));
  } else if constexpr (K <= 30) {
    t += static_cast<long long>(__float2int_rn(v)) * (1 << K);            // one IMAD.WIDE
  } else if constexpr (K == 31) {
    t += static_cast<long long>(__float2int_rn(v) * 2) * (1 << 30);
  } else {
    t += static_cast<long long>(__float2int_rn(v) * (1 << (K - 32))) << 32;
  }
}

// t rounded to nearest, |t| < 2^62, by integer arithmetic: a conversion instruction
// costs three of the FP64 unit's 64-clock slots, these about twenty-five single issue slots
__device__ __forceinline__ double to_double(long long t) {
  const unsigned long long u = t < 0 ? -static_cast<unsigned long long>(t) : static_cast<unsigned long long>(t);
  const int lz = __clzll(u);
  const unsigned long long m = u << (lz & 63);                        // bit 63 set
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);        // 53 bits, possibly carrying
  unsigned long long bits = (static_cast<unsigned long long>(1085 - lz) << 52) + r;
  bits |= static_cast<unsigned long long>(t) & 0x8000000000000000ull;
  return u != 0 ? __longlong_as_double(static_cast<long long>(bits)) : 0.0;
}

// 2^(E + k) for eb = E + 1022; NaN for eb = 0x7ff (a value that is not finite)
__device__ __forceinline__ double exp_scale(int eb, int k) {
  return eb < 0x7ff ? __hiloint2double((eb + 1 + k) << 20, 0) : __hiloint2double(0x7ff80000, 0);
}

// Steps per segment of a strip.  A segment of k steps costs about k + extra (its first
// window, its coefficients, its last results), the CTAs run one per SM: the split that
// minimises waves x (k + extra), fewest CTAs first.
inline int segment_steps(int strips, int steps, int sms, int extra) {
  long long best = -1;
  int seg = steps;
  for (int nseg = 1; nseg <= steps; ++nseg) {
    const int k = (steps + nseg - 1) / nseg, used = (steps + k - 1) / k;
    const long long waves = (static_cast<long long>(strips) * used + sms - 1) / sms, cost = waves * (k + extra);
    if (best < 0 || cost < best) {
      best = cost;
      seg = k;
    }
  }
  return seg;
}

}  // namespace dig
}  // namespace sv
