// Kernel values phi(||x - s|| / sigma) by 64-bit fixed point: the float64
// summation of the near field and of the couplings takes them from the integer
// pipes, and the float64 unit only adds up.
//
// GB300's float64 unit does 2 multiply-adds a clock on an SM; a 32 x 32 + 64
// product runs at 32 lanes a clock, adds and logic at 64 to 128 (measured).  A
// float64 Matern value at d = 8 is ~50 float64 instructions of 16 clocks a
// warp; the same value from integer products is ~58 products of one clock and
// ~100 simple instructions.
//
// Coordinates are whole multiples of 2^-F, taken from the site's float64 value
// by its bits, relative to the root box's lower corner, and split into two
// limbs X = xh 2^30 + xl.  F is chosen so that the root box's diagonal is
// below 2^59 units: a unit is at most 2^-58 of the diagonal, which is below
// the rounding of a float64 difference of two sites a unit diagonal apart.
// A pair's squared distance is the exact integer
//   T = A 2^60 + B 2^31 + C,  A = sum dh^2, B = sum dh dl, C = sum dl^2,
// one 32 x 32 + 64 product each (no carries: A < 2^58, |B| < 2^61, C < 2^64
// for d <= 16).  Then w = log2 of 1 / exp(...) with 57 fraction bits, w < 2^5,
// 2^-w by two 256-entry tables and a cubic, and phi as a float64 with all of its
// 53 bits however small it is.
//
// w < 2^5 is asked of the diagonal rounded up to a power of two (make_consts):
// a box's diagonal may be up to 11.1 to 22.2 length scales for the exponential,
// 6.4 to 12.8 for Matern-3/2 and 3.3 to 6.7 for the Gaussian, depending on where
// the diagonal lies between powers of two; larger boxes keep the float64 unit.
//
// Relative error of phi against 64-bit-mantissa arithmetic, over random and
// close pairs, d = 1..16, boxes of 1e-7 to 22 length scales, phi down to 2^-30:
// at most 1.09 2^-53, of which 1 is the rounding of the result.
#pragma once

#include <cstdint>

#include "dwfmm_internal.cuh"

namespace dw {
namespace fx {

typedef unsigned long long u64;
typedef long long s64;

constexpr int kMaxD = 16;      // C = sum dl^2 fits 64 bits
constexpr int kTable = 512;    // 2^-(j/256) 2^63, then (1 - 2^-(j/65536)) 2^64
constexpr int kQ = 57;         // fraction bits of w; w < 2^5

__host__ __device__ __forceinline__ uint32_t hi32(u64 v) { return static_cast<uint32_t>(v >> 32); }
__host__ __device__ __forceinline__ uint32_t lo32(u64 v) { return static_cast<uint32_t>(v); }
__host__ __device__ __forceinline__ u64 wide(uint32_t a, uint32_t b) { return static_cast<u64>(a) * b; }
__host__ __device__ __forceinline__ uint32_t umulhi32(uint32_t a, uint32_t b) { return hi32(wide(a, b)); }

// Top 64 bits of a * b, at most 1 unit low, for a, b <= 2^63 (the two cross
// products then add without a carry).
__host__ __device__ __forceinline__ u64 mulhi(u64 a, u64 b) {
  const u64 t = wide(lo32(a), hi32(b)) + wide(hi32(a), lo32(b));
  return wide(hi32(a), hi32(b)) + hi32(t);
}

// hi and lo parts of (hi : lo) << s, 0 <= s < 32
__host__ __device__ __forceinline__ uint32_t shl_hi(uint32_t lo, uint32_t hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
#endif
}

__host__ __device__ __forceinline__ int clz32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz(static_cast<int>(v));
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

__host__ __device__ __forceinline__ float rsqrt_seed(float x) {
#ifdef __CUDA_ARCH__
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
#else
  return 1.0f / __builtin_sqrtf(x);
#endif
}

__host__ __device__ __forceinline__ uint32_t float_bits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t u;
  __builtin_memcpy(&u, &x, 4);
  return u;
#endif
}

// sqrt(m) 2^63 for m = M 2^-64 in [1/4, 1).  With a seed y slightly below
// 1 / sqrt(m) (24 bits, unit 2^-31): g = m y, delta = 1 - g y < 2^-19 and
// sqrt(m) = g (1 - delta)^(-1/2) = g (1 + delta/2 + 3/8 delta^2 + ...); the
// next term is below 2^-58.
__host__ __device__ __forceinline__ u64 sqrt_unit(u64 M) {
  // 0.9999995 keeps y below 1 / sqrt(m) whatever the seed's rounding (2^-22)
  float y = rsqrt_seed(static_cast<float>(hi32(M))) * (65536.0f * 0.9999995f);
  y = y > 1.0f ? y : 1.0f;
  const uint32_t Y = (float_bits(y) << 8) | 0x80000000u;
  const u64 g = wide(hi32(M), Y) + hi32(wide(lo32(M), Y));              // 2^-63
  const u64 v = wide(hi32(g), Y) + hi32(wide(lo32(g), Y));              // (1 - delta) 2^62
  const u64 delta = (1ull << 62) - v;                                   // 2^-62, below 2^43
  const uint32_t dh = static_cast<uint32_t>(delta >> 11);               // 2^-51
  const u64 corr = delta + delta + umulhi32(umulhi32(dh, dh), 3u << 23);   // 2^-64
  const u64 t = wide(lo32(g), hi32(corr)) + wide(hi32(g), lo32(corr));
  return wide(hi32(g), hi32(corr)) + g + hi32(t);
}

// 2^-w for w = W 2^-57: returns 2^-f 2^63 of the fraction f and the integer
// part k < 32.  f = j1/256 + j2/65536 + f3: two table entries and
// 1 - m, m = c1 f3 - c2 f3^2 + c3 f3^3 (f3 < 2^-16, the next term is below
// 2^-69).
__host__ __device__ __forceinline__ u64 exp2_neg(u64 W, const u64* table, int& k) {
  const uint32_t wh = hi32(W), wl = lo32(W);
  k = static_cast<int>(wh >> 25);
  const u64 t1 = table[(wh >> 17) & 255u];
  const u64 d2 = table[256 + ((wh >> 9) & 255u)];
  const u64 p = t1 - mulhi(t1, d2);                                     // 2^-63
  const uint32_t fh = (wh << 23) | (wl >> 9), fl = wl << 23;            // f3 2^80
  const uint32_t u = 0x7afef7feu - umulhi32(fh, 7275u);                 // c2 - c3 f3, 2^-33
  const uint32_t x = umulhi32(umulhi32(fh, fh), u);                     // c2 f3^2 - c3 f3^3, 2^-65
  const uint32_t c1h = 0x0b17217fu, c1l = 0x7d1cf79bu;                  // ln 2, 2^-60
  const u64 m = wide(fh, c1h) + hi32(wide(fh, c1l) + wide(fl, c1h)) -
                static_cast<u64>(static_cast<s64>(static_cast<int32_t>(x)) * 2048);   // 2^-76
  return p - (mulhi(p, m) >> 12);
}

// m 2^e 2^-52 for m in [2^52, 2^53].
__host__ __device__ __forceinline__ double from_bits(u64 m, int e) {
  const u64 b = m + (static_cast<u64>(static_cast<uint32_t>(e + 1022)) << 52);   // m carries 1 into the exponent
#ifdef __CUDA_ARCH__
  return __longlong_as_double(static_cast<s64>(b));
#else
  double v;
  __builtin_memcpy(&v, &b, 8);
  return v;
#endif
}

// phi from T = A 2^60 + B 2^31 + C (pairs of one tree: T < 2^118), for P
// independent pairs side by side: one chain of dependent products is too long
// for the warps that fit.
template <int KER, int P>
__host__ __device__ __forceinline__ void phi64(const u64 (&A)[P], const s64 (&B)[P], const u64 (&C)[P], const Consts& c,
                                               const u64* table, double (&out)[P]) {
  u64 W[P];
  if (KER == DWFMM_K_GAUSS) {
    // T 2^-55 in 63 bits; + 1 because the two floors may add up to -1
#pragma unroll
    for (int q = 0; q < P; ++q) W[q] = mulhi((A[q] << 5) + static_cast<u64>(B[q] >> 24) + (C[q] >> 55) + 1, c.K);
  } else {
    // T 2^-32 in three words (+ 1: the two floors may add up to -1); below
    // 2^64 (a distance under 2^-11 of the diagonal) all of T, shifted up, so
    // that the root keeps its bits
    uint32_t w3[P], w2[P], w1[P];
    int h[P];
    bool close = false;
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const u64 low = static_cast<u64>(lo32(A[q]) << 28) + lo32(static_cast<u64>(B[q] >> 1)) + hi32(C[q]) + 1;
      const u64 top = (A[q] >> 4) + static_cast<u64>(B[q] >> 33) + hi32(low);
      w3[q] = hi32(top);
      w2[q] = lo32(top);
      w1[q] = lo32(low);
      h[q] = -5;
      close |= w3[q] == 0;
    }
    if (close) {
#pragma unroll
      for (int q = 0; q < P; ++q) {
        if (w3[q] != 0) continue;
        const u64 lo1 = C[q] + (static_cast<u64>(B[q]) << 31), lo = lo1 + (A[q] << 60);
        w3[q] = lo32((A[q] >> 4) + static_cast<u64>(B[q] >> 33) + (lo1 < C[q] ? 1u : 0u) + (lo < lo1 ? 1u : 0u));
        w2[q] = hi32(lo);
        w1[q] = lo32(lo) | 1u;
        h[q] = 11;
        for (int z = 0; z < 2 && w3[q] == 0; ++z) {
          w3[q] = w2[q];
          w2[q] = w1[q];
          w1[q] = 0;
          h[q] += 16;
        }
      }
    }
    u64 M[P];
#pragma unroll
    for (int q = 0; q < P; ++q) {
      const int s = clz32(w3[q]) & ~1;
      M[q] = (static_cast<u64>(shl_hi(w2[q], w3[q], s)) << 32) | shl_hi(w1[q], w2[q], s);
      h[q] += s >> 1;
    }
    // sqrt(T) = sqrt_unit 2^(1 - h - s/2), s >= 10 as T < 2^118
#pragma unroll
    for (int q = 0; q < P; ++q) W[q] = mulhi(sqrt_unit(M[q]), c.K) >> h[q];
  }
#pragma unroll
  for (int q = 0; q < P; ++q) {
    int k;
    u64 e = exp2_neg(W[q], table, k);
    if (KER == DWFMM_K_MATERN32) {
      // (1 + t) e^-t, t = w ln 2, 1 + t < 2^5
      const u64 t = mulhi(W[q], 0xb17217f7d1cf79acull);                   // 2^-57 (W < 2^62: no carry either)
      e = mulhi(e, t + t + ((1ull << 58) + 1));                           // phi 2^k 2^57, in (2^56, 2^62)
      const int s = clz32(hi32(e)) - 1;
      out[q] = from_bits(((e << s) + 512) >> 10, 5 - s - k);
    } else {
      out[q] = from_bits((e + 512) >> 10, -1 - k);                        // e in (2^62, 2^63]
    }
  }
}

// x in units of 2^-F, modulo 2^64, rounded to nearest (ties up): from the
// float64's bits, exact whenever x is a multiple of the unit.
__host__ __device__ __forceinline__ u64 to_units(double x, int F) {
#ifdef __CUDA_ARCH__
  const u64 b = static_cast<u64>(__double_as_longlong(x));
#else
  u64 b;
  __builtin_memcpy(&b, &x, 8);
#endif
  const int e = static_cast<int>((b >> 52) & 0x7ff);
  u64 m = b & 0xfffffffffffffull;
  if (e) m |= 1ull << 52;
  const int s = (e ? e : 1) - 1075 + F;
  u64 v;
  if (s >= 64) v = 0;
  else if (s >= 0) v = m << s;
  else if (s > -64) v = ((m >> (-s - 1)) + 1) >> 1;
  else v = 0;
  return (b >> 63) ? 0ull - v : v;
}

// ---- constants of a tree (host) -------------------------------------------

// The table of exp2_neg: Taylor series of exp(-j ln2 / 256) and
// exp(-j ln2 / 65536) with 100 fraction bits.
inline void make_table(u64* t) {
  typedef unsigned __int128 u128;
  const u64 ln2 = 0xb17217f7d1cf79acull;   // 2^-64
  for (int j = 0; j < kTable; ++j) {
    const u128 x = static_cast<u128>(ln2) * static_cast<unsigned>(j & 255);   // 2^-72 or 2^-80
    const u64 xl = static_cast<u64>(j < 256 ? x >> 8 : x >> 16);              // 2^-64
    u128 term = static_cast<u128>(1) << 100, sum = term;
    for (unsigned n = 1; n < 30; ++n) {
      const u64 th = static_cast<u64>(term >> 64), tl = static_cast<u64>(term);
      term = (static_cast<u128>(th) * xl + ((static_cast<u128>(tl) * xl) >> 64)) / n;
      if (n & 1) sum -= term;
      else sum += term;
    }
    if (j < 256) t[j] = static_cast<u64>((sum + (static_cast<u128>(1) << 36)) >> 37);
    else t[j] = static_cast<u64>(((static_cast<u128>(1) << 100) - sum + (static_cast<u128>(1) << 35)) >> 36);
  }
}

// Positive value hi 2^e with a 64-bit mantissa (top bit set).
struct Big {
  u64 m;
  int e;
};

// N / v for a 128-bit numerator N 2^en (top bit set).
inline Big big_div(unsigned __int128 n, int en, double v) {
  int ev;
  const u64 mv = static_cast<u64>(__builtin_ldexp(__builtin_frexp(v, &ev), 53));   // v = mv 2^(ev - 53), 53 bits
  unsigned __int128 q = n / mv;   // at least 75 bits
  int e = en - (ev - 53);
  while (q >> 64) {
    q >>= 1;
    ++e;
  }
  return Big{static_cast<u64>(q), e};
}

// Scale of w for a box whose diagonal is below 2^(59 - F); false when w may
// reach 2^5 at that bound.
inline bool make_consts(int kernel, double sigma, int F, Consts& c) {
  typedef unsigned __int128 u128;
  const u128 log2e = (static_cast<u128>(0xb8aa3b295c17f0bbull) << 64) | 0xbe87fed0691d3e89ull;     // 2^-127
  const u128 s3log2e = (static_cast<u128>(0x9fecaf61323924e0ull) << 64) | 0xcaa2da66044631f5ull;   // 2^-126
  Big b;
  int e;   // w 2^57 = (T 2^-55 or sqrt(T) 2^(63 - 59)) K 2^-64, K = b.m 2^e
  if (kernel == DWFMM_K_GAUSS) {
    const Big h = big_div(log2e, -128, sigma);   // log2(e) / (2 sigma)
    b = big_div(static_cast<u128>(h.m) << 64, h.e - 64, sigma);
    e = b.e - 2 * F + 55 + 64 + kQ;
  } else {
    b = kernel == DWFMM_K_EXP ? big_div(log2e, -127, sigma) : big_div(s3log2e, -126, sigma);
    e = b.e - F - 4 + 64 + kQ;
  }
  // K <= 2^63 keeps w below 2^5
  c.K = e <= -64 ? 0 : e < 0 ? b.m >> -e : 0;
  return e < 0;
}

// Largest F with diag 2^F < 2^59.
inline int units_exponent(double diag) {
  int e;
  (void)__builtin_frexp(diag, &e);   // diag < 2^e
  return 59 - e;
}

}  // namespace fx
}  // namespace dw
