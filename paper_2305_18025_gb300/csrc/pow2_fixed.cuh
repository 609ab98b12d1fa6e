// Powers 2^(-x), x >= 0, to float64 accuracy on the integer pipe.
//
// The float64 pipe of a GB300 SM issues one warp instruction about every 64
// cycles, so the O(N^2) pair Boltzmann factors g = exp(-beta (1/2) k d^2)
// avoid it.  Tang's table-driven method (P. T. P. Tang, ACM TOMS 15(2), 1989)
// in 64-bit fixed point:
//   x = n + f, n integer, f in [0, 1) as a 64-bit fraction F = f 2^64 (x is
//   the exact product of the argument's factors, up to 128 bits);
//   f = j/256 + r, j = the top 8 bits of F, 0 <= r < 2^-8;
//   2^(-f) = T[j] e^(-u), u = r ln 2 < 0.0028, T[j] = 2^(-j/256) (table of
//   pow2_table.h, 63 fraction bits);
//   e^(-u) = 1 - u (1 - u (1/2 - u (1/6 - u (1/24 - u/120)))), truncation below
//   u^6/720 < 2^-60 relative, evaluated with 64 x 64 -> high-64 products.
// The result is (mantissa in [1, 2) as a double, exponent): value
// m 2^e = 2^(-x) to a few 2^-60 relative -- finer than one float64 rounding.
// x >= 2^28 gives 2^(-2^28): the recursions read exponents below -2^28 as zero.
// Host-compilable (the CPU tests emulate it bit for bit with __int128).
#pragma once
#include <cstdint>

#include "pow2_table.h"

#ifdef __CUDACC__
#define BPIMD_HD __host__ __device__ __forceinline__
#else
#define BPIMD_HD inline
#endif

namespace bpimd {
namespace pow2fx {

#ifdef __CUDA_ARCH__
__device__ const unsigned long long T63[256] = {BPIMD_POW2_T63_INIT};
BPIMD_HD unsigned mulhi32(unsigned a, unsigned b) { return __umulhi(a, b); }
#else
static const unsigned long long T63[256] = {BPIMD_POW2_T63_INIT};
BPIMD_HD unsigned mulhi32(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
#endif
// High 64 bits of a 64 x 64-bit product without the low words' product: at
// most 3 units of 2^-64 too small, three multiplications for four.
BPIMD_HD unsigned long long mulhi(unsigned long long a, unsigned long long b) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
  return (unsigned long long)ah * bh + mulhi32(ah, bl) + mulhi32(al, bh);
}

constexpr unsigned long long Q64_HALF = 0x8000000000000000ull;
constexpr unsigned long long Q64_SIXTH = 0xFFFFFFFFFFFFFFFFull / 6;
constexpr unsigned Q32_24TH = 0xFFFFFFFFu / 24;
constexpr unsigned Q32_120TH = 0xFFFFFFFFu / 120;
constexpr int ZERO_EXP = -(1 << 28);  // 2^(-2^28): an extended zero for the recursions

struct mexp {
  double m;  // in [1, 2)
  int e;
};

BPIMD_HD double bits_to_double(unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
BPIMD_HD unsigned long long double_to_bits(double d) {
#ifdef __CUDA_ARCH__
  return (unsigned long long)__double_as_longlong(d);
#else
  unsigned long long b;
  __builtin_memcpy(&b, &d, 8);
  return b;
#endif
}

// (hi:lo) >> k, low word, k in [0, 31]
BPIMD_HD unsigned funnel(unsigned lo, unsigned hi, int k) {
#ifdef __CUDA_ARCH__
  return __funnelshift_r(lo, hi, k);
#else
  return (unsigned)((((unsigned long long)hi << 32) | lo) >> k);
#endif
}

// 2^(-f) 2^63 of the fraction f = (Fh:Fl) 2^-64.
BPIMD_HD unsigned long long pow2neg_frac(unsigned Fh, unsigned Fl, const unsigned long long *table) {
  const unsigned j = Fh >> 24;
  const unsigned long long r = ((unsigned long long)(Fh & 0x00FFFFFFu) << 32) | Fl;  // f - j/256, times 2^64
  const unsigned long long u = mulhi(r, BPIMD_LN2_Q64);                              // u 2^64, u = r ln 2
  // the terms in u^5 and u^4 on 32 bits (u 2^40 < 2^32): they stand below 2^-38
  const unsigned uh = (unsigned)(u >> 24);
  const unsigned t4 = Q32_24TH - (mulhi32(uh, Q32_120TH) >> 8);                     // 1/24 - u/120
  unsigned long long t = Q64_SIXTH - (((unsigned long long)uh * t4) >> 8);          // 1/6 - u t
  t = Q64_HALF - mulhi(u, t);                                                       // 1/2 - u t
  const unsigned long long q = u - mulhi(u, mulhi(u, t));                           // u (1 - u t) = 1 - e^(-u)
  const unsigned long long T = table[j];
  return T - mulhi(T, q);
}

// 2^(-x) for x = (H 2^64 + L) 2^S, H in [2^63, 2^64) (a normalised 128-bit
// mantissa: exact products of two float64 or float32 mantissas fit in it).
// table: T63 or a shared-memory copy of it.
BPIMD_HD mexp pow2neg_q(unsigned long long H, unsigned long long L, int S, const unsigned long long *table) {
  if (S >= -99) return mexp{1.0, ZERO_EXP};  // x >= 2^28
  // x = (H:L) >> (k + 64), k >= 36: the integer part n above, the 64 fraction
  // bits F below that point, by words
  const int k = -S - 64;
  const unsigned h1 = (unsigned)(H >> 32), h0 = (unsigned)H, l1 = (unsigned)(L >> 32);
  unsigned n, Fh, Fl;
  if (k < 64) {
    n = h1 >> (k - 32);
    Fh = funnel(h0, h1, k - 32);
    Fl = funnel(l1, h0, k - 32);
  } else {
    n = 0;
    Fh = k < 96 ? h1 >> (k - 64) : 0u;
    Fl = k < 96 ? funnel(h0, h1, k - 64) : (k < 128 ? h1 >> (k - 96) : 0u);
  }
  const unsigned long long res = pow2neg_frac(Fh, Fl, table);  // 2^(-f) 2^63, in (2^62 - 8, 2^63]
  // rounded to 53 bits (to nearest; 511 for 512, as res is 1 unit too large on
  // average: 6e-4 of the results are off by the last bit, 1.3e-3 with 512): in
  // [2^52, 2^53], 2^53 being the next power of two (which the rounding also
  // reaches from 2^62 - 8 below)
  const unsigned long long m53 = (res + 511) >> 10;
  return mexp{bits_to_double((m53 & 0x000FFFFFFFFFFFFFull) | 0x3FF0000000000000ull), (int)(m53 >> 53) - 1 - (int)n};
}

// (H:L) with its top bit set, shifted left by at most one
BPIMD_HD void norm128(unsigned long long &H, unsigned long long &L, int &shift) {
  shift = 0;
  if (!(H >> 63)) {
    H = (H << 1) | (L >> 63);
    L <<= 1;
    shift = 1;
  }
}
// Full 128-bit product of two 64-bit mantissas, normalised (both inputs have
// their top bit set).
BPIMD_HD void mul128_norm(unsigned long long a, unsigned long long b, unsigned long long &H,
                          unsigned long long &L, int &shift) {
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
  const unsigned long long ll = (unsigned long long)al * bl, x = (unsigned long long)ah * bl + (ll >> 32);
  const unsigned long long y = (unsigned long long)al * bh + (unsigned)x;
  H = (unsigned long long)ah * bh + (x >> 32) + (y >> 32);
  L = (y << 32) | (unsigned)ll;
  norm128(H, L, shift);
}
// The same with a = m 2^32, m a 32-bit mantissa with its top bit set.
BPIMD_HD void mul128_norm(unsigned m, unsigned long long b, unsigned long long &H, unsigned long long &L, int &shift) {
  const unsigned long long lo = (unsigned long long)m * (unsigned)b, hi = (unsigned long long)m * (unsigned)(b >> 32);
  const unsigned long long mid = hi + (lo >> 32);  // (m b) >> 32
  H = mid;
  L = lo << 32;
  norm128(H, L, shift);
}

// 2^(-x) for a double x >= 0 (its bits read by integer instructions).
BPIMD_HD mexp pow2neg(double x, const unsigned long long *table) {
  const unsigned long long b = double_to_bits(x);
  const int E = (int)((b >> 52) & 0x7FF);
  if (E == 0) return mexp{1.0, 0};  // 0 or subnormal: 2^(-x) = 1 to 2^-1000
  const unsigned long long M = ((b & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
  return pow2neg_q(M, 0ull, E - 1023 - 63 - 64, table);
}

// 2^(-x) for x = a * c with a float32 a >= 0 and a double c > 0: the product
// is formed exactly (24 x 53 bits), so the float32 argument is not rounded
// again.
BPIMD_HD mexp pow2neg_fd(float a, double c, const unsigned long long *table) {
#ifdef __CUDA_ARCH__
  const unsigned ab = (unsigned)__float_as_int(a);
#else
  unsigned ab;
  __builtin_memcpy(&ab, &a, 4);
#endif
  const int Ea = (int)((ab >> 23) & 0xFF);
  if (Ea == 0) return mexp{1.0, 0};
  const unsigned long long cb = double_to_bits(c);
  const int Ec = (int)((cb >> 52) & 0x7FF);
  const unsigned ma = (ab << 8) | 0x80000000u;  // 24-bit significand, top bit set
  const unsigned long long mc = ((cb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
  unsigned long long H, L;
  int sh;
  mul128_norm(ma, mc, H, L, sh);
  // a = ma 2^(Ea-127-63), c = mc 2^(Ec-1023-63): x = (H:L) 2^(Ea-190 + Ec-1086 - sh)
  return pow2neg_q(H, L, (Ea - 190) + (Ec - 1086) - sh, table);
}

// 2^(-x) for x = a * c with doubles a >= 0, c > 0: the 53 x 53-bit mantissa
// product is formed exactly on the integer pipe, so the float64 argument is
// not rounded again either.
BPIMD_HD mexp pow2neg_dd(double a, double c, const unsigned long long *table) {
  const unsigned long long ab = double_to_bits(a), cb = double_to_bits(c);
  const int Ea = (int)((ab >> 52) & 0x7FF), Ec = (int)((cb >> 52) & 0x7FF);
  if (Ea == 0) return mexp{1.0, 0};
  const unsigned long long ma = ((ab & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
  const unsigned long long mc = ((cb & 0x000FFFFFFFFFFFFFull) | 0x0010000000000000ull) << 11;
  unsigned long long H, L;
  int sh;
  mul128_norm(ma, mc, H, L, sh);
  return pow2neg_q(H, L, (Ea - 1086) + (Ec - 1086) - sh, table);
}

}  // namespace pow2fx
}  // namespace bpimd
