// Molecular dynamics of the bosonic ring polymers.
//
// The paper samples exp(-beta (V^{[1,N]} + U-bar)) (Eq.
// int-of-sum-all-permutations; spring frequency w_P = sqrt(P)/(beta hbar),
// Eq. eperm; U-bar = (1/P) sum_j U(r_1^j..r_N^j)) with molecular dynamics and
// a thermostat, without stating the integrator.  This file runs Cartesian
// BAOAB Langevin steps at temperature kT (default 1/beta) with bead mass m:
//   B  v += (dt/2) F/m            A  x += (dt/2) v
//   O  v  = c1 v + c2 z,  c1 = exp(-gamma dt), c2 = sqrt((1 - c1^2) kT/m)
//   A  x += (dt/2) v              F = -grad(V^{[1,N]} + U-bar)(x)
//   B  v += (dt/2) F/m
// with U = sum_l (1/2) m w0^2 |r_l|^2 (harmonic trap) + sum_{l<l'} g
// exp(-|r_l - r_l'|^2 / (2 s^2)) (Gaussian repulsion) or Lennard-Jones
// 4 eps ((sig/r)^12 - (sig/r)^6) truncated and shifted at rc (liquid helium;
// cell lists in pairs.cu when the box holds >= 3 cutoffs per side) between
// beads of equal index; in a periodic box every spring and pair uses the
// minimum image.  The exchange force is one evaluation of Algorithm 1 (the kernels of
// prep.cu, chain.cu, force.cu).
//
// Thermostat noise: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11),
// written here from its published definition.  Element e = 4g + i of the
// velocity array at step s takes word i of the block with counter
// (g, s mod 2^32, s div 2^32, 0) and key (seed mod 2^32, seed div 2^32);
// words become uniforms u = (x + 1/2) 2^-32 and pairs of uniforms become
// normals by the Box-Muller transform (float64; MIXED: float32).
//
// A step's closing B and the next step's B A O A are one kernel.  The physical
// force and the next step's noise need the positions and the counter only, so
// they are formed while the recursions run.  One step is captured once into a
// CUDA graph bound to the caller's position and velocity buffers and replayed;
// the step counter lives in device memory and is advanced by the closing B.
#include <cmath>
#include <vector>
#include <type_traits>

#include "context.cuh"
#include "pairg.cuh"
#include "pairs.cuh"

namespace bpimd {
namespace {

constexpr int MD_THREADS = 256;
constexpr int ENERGY_THREADS = 1024;  // the one block that adds a call's partial energies
constexpr int EXT_THREADS = 128;
constexpr int EXT_WARPS = EXT_THREADS / 32;
// particles a thread and lanes a particle in the all-pairs force: float64 pairs
// take ~15 times as long, and the smaller blocks spread them evenly (in a box,
// N = 512, P = 32, four steps: Gaussian 2131 us and Lennard-Jones 4217 with one
// particle and eight lanes; two and eight 2563, 5152; one and four 2520, 5117)
constexpr int ext_ppt(bool mixed) { return mixed ? 2 : 1; }
constexpr int ext_split(bool mixed) { return mixed ? 4 : 8; }
constexpr int ext_particles(bool mixed) { return ext_ppt(mixed) * EXT_THREADS / ext_split(mixed); }
constexpr int EXT_CHUNK = 1024;  // positions of one bead index staged per pass

struct Dbl3 {
  double x, y, z;
};

__device__ __forceinline__ void philox4x32_10(uint32_t c[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint32_t lo0 = 0xD2511F53u * c[0], hi0 = __umulhi(0xD2511F53u, c[0]);
    const uint32_t lo1 = 0xCD9E8D57u * c[2], hi1 = __umulhi(0xCD9E8D57u, c[2]);
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
}

template <bool MIXED>
__device__ __forceinline__ void box_muller(const uint32_t x[4], double z[4]) {
  if (MIXED) {
    float u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = ((float)x[i] + 0.5f) * 2.3283064365386963e-10f;
    const float ra = sqrtf(-2.0f * logf(u[0])), rb = sqrtf(-2.0f * logf(u[2]));
    float sa, ca, sb, cb;
    sincosf(6.28318530717958648f * u[1], &sa, &ca);
    sincosf(6.28318530717958648f * u[3], &sb, &cb);
    z[0] = ra * ca; z[1] = ra * sa; z[2] = rb * cb; z[3] = rb * sb;
  } else {
    double u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) u[i] = ((double)x[i] + 0.5) * 2.3283064365386962890625e-10;
    const double two_pi = 6.283185307179586476925286766559;
    const double ra = sqrt(-2.0 * log(u[0])), rb = sqrt(-2.0 * log(u[2]));
    double sa, ca, sb, cb;
    sincos(two_pi * u[1], &sa, &ca);
    sincos(two_pi * u[3], &sb, &cb);
    z[0] = ra * ca; z[1] = ra * sa; z[2] = rb * cb; z[3] = rb * sb;
  }
}

// Thermostat kicks c2 z of elements 4g .. 4g+3 (one Philox block) of step s.
// They depend on the counter only, so the pair-force kernel's spare blocks
// form them while the recursions run (a float64 Box-Muller is ~15 us of
// latency on the step's path otherwise).
template <bool MIXED>
__device__ __forceinline__ void thermostat_kicks(long long g, unsigned long long s, uint32_t k0, uint32_t k1,
                                                 double (&z)[4]) {
  uint32_t c[4] = {(uint32_t)g, (uint32_t)s, (uint32_t)(s >> 32), 0u};
  philox4x32_10(c, k0, k1);
  box_muller<MIXED>(c, z);
}

// K: closing B of a step (and its counter); A: B A O of the next, with the
// full force F + Fx (exchange, physical) and the thermostat kicks zc (null:
// none).  Two elements a thread, 16-byte accesses.
template <bool K, bool A>
__global__ void __launch_bounds__(MD_THREADS) md_update_kernel(double *__restrict__ x, double *__restrict__ v,
                                                               const double *__restrict__ F,
                                                               const double *__restrict__ Fx,
                                                               const double *__restrict__ zc, long long n, double h,
                                                               double half_dt, double c1, unsigned long long *step) {
  pdl_wait();
  auto one = [&](double &xe, double &ve, double Fe, double ze) {
    if (K) ve = fma(h, Fe, ve);  // B
    if (A) {
      ve = fma(h, Fe, ve);        // B
      xe = fma(half_dt, ve, xe);  // A
      ve = fma(c1, ve, ze);       // O
      xe = fma(half_dt, ve, xe);  // A
    }
  };
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; 2 * g < n; g += stride) {
    if (2 * g + 1 < n) {
      const double2 f = ((const double2 *)F)[g], fx = ((const double2 *)Fx)[g];
      const double2 z = A && zc ? ((const double2 *)zc)[g] : make_double2(0.0, 0.0);
      double2 ve = ((double2 *)v)[g], xe = A ? ((double2 *)x)[g] : make_double2(0.0, 0.0);
      one(xe.x, ve.x, f.x + fx.x, z.x);
      one(xe.y, ve.y, f.y + fx.y, z.y);
      if (A) ((double2 *)x)[g] = xe;
      ((double2 *)v)[g] = ve;
    } else {
      const long long e = 2 * g;
      double xe = A ? x[e] : 0.0, ve = v[e];
      one(xe, ve, F[e] + Fx[e], A && zc ? zc[e] : 0.0);
      if (A) x[e] = xe;
      v[e] = ve;
    }
  }
  if (K && blockIdx.x == 0 && threadIdx.x == 0) *step += 1ull;
}

// m 2^e of the integer-pipe power of two as a double (e <= 0; the exponent is
// added with integer instructions; results below the normal range give 0)
__device__ __forceinline__ double pow2_value(pow2fx::mexp r) {
  const long long b = __double_as_longlong(r.m);
  return ((int)(b >> 52) + r.e <= 0) ? 0.0 : __longlong_as_double(b + ((long long)r.e << 52));
}

// float64 -> float32, round to nearest even, on the integer pipe (a
// conversion instruction runs on GB300's narrow float64 pipe); results below
// the float32 normal range flush to a signed zero, so the value must be
// finite and below 2^128 in magnitude.  Bit-identical to __double2float_rn
// for every normal float32 result.
__device__ __forceinline__ float f32_of_f64(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const unsigned sign = (unsigned)(b >> 32) & 0x80000000u;
  const int ex = (int)((b >> 52) & 0x7ff) - 1023 + 127;
  const unsigned long long m = b & 0xFFFFFFFFFFFFFull;
  unsigned r = (unsigned)(m >> 29);
  const unsigned long long rem = m & ((1ull << 29) - 1);
  r += (rem > (1ull << 28)) || (rem == (1ull << 28) && (r & 1u));
  return ex <= 0 ? __uint_as_float(sign) : __uint_as_float(sign | (((unsigned)ex << 23) + r));
}

// float32 -> float64 on the integer pipe (exact; zero and subnormal inputs give
// a signed zero; the value must be finite)
__device__ __forceinline__ double f64_of_f32(float x) {
  const unsigned b = __float_as_uint(x);
  const unsigned ex = (b >> 23) & 0xffu;
  const unsigned long long s = (unsigned long long)(b & 0x80000000u) << 32;
  if (ex == 0) return __longlong_as_double((long long)s);
  return __longlong_as_double(
      (long long)(s | ((unsigned long long)(ex - 127 + 1023) << 52) | ((unsigned long long)(b & 0x7fffffu) << 29)));
}

// Deterministic block sum (fixed shuffle tree, then warps in order); thread 0 gets it.
__device__ __forceinline__ double block_sum(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) s += red[q];
  __syncthreads();
  return s;
}

// --------------------------------- float64 Gaussian pairs on integer mantissas
// GB300's float64 pipe takes ~75 cycles a warp instruction, and a directed pair
// in float64 needs ten of them beside the integer power of two.  Here it forms
// the three differences only.  Every later quantity keeps a mantissa and an
// exponent of its own, so that a pair is as accurate relative to itself as in
// float64, however near, far, wide or flat the system is: the squares are summed
// on the scale of the largest component (2^-57 of d^2), times log2(e)/(2 s^2)
// they are the argument of the power of two (2^-60), and e d is added to 96-bit
// sums whose unit lies 62 bits below their largest term.  A pair is ~260
// instructions, mostly of the integer pipe, beside the float64 pipe's ~57 cycles:
// 408 us a pass at N = 1024, P = 32 (455 with e d multiplied and summed in float64,
// ~720 all in float64).  One particle a thread: with two (122 registers for 80)
// the pass took 460 us.
struct Acc96 {  // (hi:mid:lo) 2^(B - 94), hi signed
  unsigned lo, mid, hi;
  int B;
};
struct Sum96 {
  unsigned lo, mid, hi;
};
__device__ __forceinline__ void add_words(unsigned &lo, unsigned &mid, unsigned &hi, unsigned x, unsigned y, unsigned z) {
  asm("add.cc.u32 %0, %0, %3;\n addc.cc.u32 %1, %1, %4;\n addc.u32 %2, %2, %5;"
      : "+r"(lo), "+r"(mid), "+r"(hi)
      : "r"(x), "r"(y), "r"(z));
}
// (hi:mid:lo) as a signed integer, rounded to float64
__device__ __forceinline__ double value96(unsigned lo, unsigned mid, unsigned hi) {
  const long long top = (long long)(((unsigned long long)hi << 32) | mid);
  return fma((double)top, 4294967296.0, (double)lo);
}
// Room for a term of exponent pe: it is placed 31 bits below the sum's sign,
// and later ones up to 2^16 times as large need no other move.
constexpr int ACC_EMPTY = -(1 << 24), ACC_ROOM = 15;  // 2^13 terms a lane stay below 2^(95 - 2)
__device__ __forceinline__ void acc_raise(Acc96 &a, int pe) {
  int r = pe + 31 - a.B;
  a.B = pe + 31;
  if (r > 96) r = 96;
  for (; r > 0; r -= 31) {
    const int t = min(r, 31);
    a.lo = __funnelshift_r(a.lo, a.mid, t);
    a.mid = __funnelshift_r(a.mid, a.hi, t);
    a.hi = (unsigned)((int)a.hi >> t);
  }
}
// a += P 2^(pe - 62), |P| < 2^63, s = a.B - pe >= ACC_ROOM
__device__ __forceinline__ void acc_add(Acc96 &a, long long P, int s) {
  const long long top = P >> min(s, 63);
  const unsigned low = s < 32 ? __funnelshift_r(0u, (unsigned)P, s) : (unsigned)(P >> min(s - 32, 63));
  add_words(a.lo, a.mid, a.hi, low, (unsigned)top, (unsigned)((unsigned long long)top >> 32));
}
__device__ __forceinline__ double acc_value(const Acc96 &a) {
  const int k = max(a.B - 94, -2044), k1 = k >> 1;  // in two factors: either is a normal number
  const double v = value96(a.lo, a.mid, a.hi) * __longlong_as_double((long long)(k1 + 1023) << 52) *
                   __longlong_as_double((long long)(k - k1 + 1023) << 52);
  return fabs(v) < 1e-300 ? 0.0 : v;  // zero differences, each counted as 2^-1023
}

struct GaussSum {  // sums over a lane's partners
  Acc96 f[3];      // e d
  Sum96 u;         // e, 2^-62 (the particle's own e = 1 included)
  int bad;         // components that met a non-finite difference
};

// One directed pair of difference d: adds e d and e, e = 2^(-g2c |d|^2).
__device__ __forceinline__ void gauss_pair(const double (&d)[3], unsigned long long gm, int ge,
                                           const unsigned long long *T63, GaussSum &a) {
  unsigned long long M[3];  // |d| = M 2^(ef - 1023 - 63), M in [2^63, 2^64); a zero counts as 2^-1023
  int ef[3], sg[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(d[c]);
    const int hi = (int)(b >> 32);
    sg[c] = hi >> 31;
    ef[c] = (hi >> 20) & 0x7ff;
    M[c] = (b << 11) | (1ull << 63);
  }
  const int em = max(ef[0], max(ef[1], ef[2]));
  if (em == 0x7ff) {
#pragma unroll
    for (int c = 0; c < 3; ++c) a.bad |= (ef[c] == 0x7ff) << c;
  }
  // |d|^2 = (q + w 2^-31) 2^(2 (em - 1023) - 58); the low words' squares and the
  // cuts amount to two units on average, with which q starts: 2^-60 rms, no mean error
  unsigned long long q = 2, w = 0;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const unsigned long long A = M[c] >> (min(em - ef[c], 61) + 2);
    const unsigned h = (unsigned)(A >> 32), l = (unsigned)A;
    q += (unsigned long long)h * h;
    w += (unsigned long long)h * l;
  }
  const unsigned long long Y = pow2fx::mulhi((q + (w >> 31)) << 2, gm);  // g2c |d|^2 = Y 2^-s
  const int s = 59 - ge - 2 * (em - 1023);
  const bool far = s < 49;  // Y >= 2^59: e < 2^-1024, as a float64 e would be zero
  const bool whole = s < 64;
  const unsigned long long F = whole ? Y << ((64 - s) & 63) : Y >> min(s - 64, 63);
  const int n = whole ? (int)(Y >> (s & 63)) : 0;
  const unsigned long long res = far ? 0ull : pow2fx::pow2neg_frac((unsigned)(F >> 32), (unsigned)F, T63);
  const unsigned long long e = (unsigned)n > 62u ? 0ull : res >> (n + 1);
  add_words(a.u.lo, a.u.mid, a.u.hi, (unsigned)e, (unsigned)(e >> 32), 0u);
  if (far) return;
  const int pe = -1023 - n;
  if (min(a.f[0].B - ef[0], min(a.f[1].B - ef[1], a.f[2].B - ef[2])) - pe < ACC_ROOM) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      if (a.f[c].B - ef[c] - pe < ACC_ROOM) acc_raise(a.f[c], ef[c] + pe);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const long long P = (long long)pow2fx::mulhi(res, M[c]);
    acc_add(a.f[c], (P ^ (long long)sg[c]) - (long long)sg[c], a.f[c].B - ef[c] - pe);
  }
}

// Two float32 numbers in one 64-bit register: one instruction issued for two
// IEEE operations (rounded as the scalar ones).
using F2 = unsigned long long;
__device__ __forceinline__ F2 pack2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(F2 v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// -grad U-bar into Fx, per bead index j and block of PPT * 128 / SPLIT particles
// (all pairs).  The SPLIT lanes of a thread group take the partners q = sub,
// sub + SPLIT, ... of each staged chunk for PPT particles each, and combine their
// sums by a fixed shuffle butterfly; U-bar partial sum per block.  Two particles a
// thread (half the block apart) where a load from shared memory counts: it serves
// two pairs then (a 16-byte load a pair kept the shared-memory pipe at 79 % of its
// rate, 23.6 instructions a pair).
// The positions of bead j of all particles pass through shared memory in chunks.
// Pairs: Gaussian g exp(-r^2/(2 s^2)), or Lennard-Jones 4 eps ((sig/r)^12 -
// (sig/r)^6) truncated and shifted at rc; in a periodic box (PBC) pair distances
// by minimum image.  MIXED: pair terms in float32, accumulated per lane in float32.
template <bool MIXED, bool PBC, int SPLIT, int PPT>
__device__ __forceinline__ double ext_force_body(const double *__restrict__ pos, double *__restrict__ Fx, int N,
                                                 int P, const PairParams &pp, int lb, int j,
                                                 typename std::conditional<MIXED, float4, Dbl3>::type *sr,
                                                 double *red, unsigned long long *T63s) {
  using R = typename std::conditional<MIXED, float, double>::type;
  using R4 = typename std::conditional<MIXED, float4, Dbl3>::type;
  constexpr int HALF = EXT_THREADS / SPLIT;  // particles of a block: PPT HALF
  const int sub = threadIdx.x % SPLIT;
  int l[PPT];
  double rd[PPT][3];
  R px[PPT], py[PPT], pz[PPT];
#pragma unroll
  for (int h = 0; h < PPT; ++h) {
    l[h] = lb * PPT * HALF + h * HALF + threadIdx.x / SPLIT;
    const double *r = pos + ((size_t)min(l[h], N - 1) * P + j) * 3;
    rd[h][0] = r[0]; rd[h][1] = r[1]; rd[h][2] = r[2];
    // mixed: float32 positions and constants from integer-pipe conversions
    // and host-formed copies (no float64 work)
    if constexpr (MIXED) { px[h] = f32_of_f64(r[0]); py[h] = f32_of_f64(r[1]); pz[h] = f32_of_f64(r[2]); }
    else { px[h] = r[0]; py[h] = r[1]; pz[h] = r[2]; }
  }
  R a, L, invL, sig2, rc2;
  if constexpr (MIXED) { a = pp.fa; L = pp.fL; invL = pp.finvL; sig2 = pp.fsig2; rc2 = pp.frc2; }
  else { a = -0.5 * pp.inv_s2; L = pp.L; invL = pp.invL; sig2 = pp.sig2; rc2 = pp.rc2; }
  if (!MIXED) pairg::table_init(T63s);  // float64: the integer-pipe power of two (read after the first barrier)
  auto img = [&](R d) -> R {
    if constexpr (PBC) return d - L * (MIXED ? (R)rintf((float)(d * invL)) : (R)rint((double)(d * invL)));
    else return d;
  };
  constexpr bool INTEGER = !MIXED && !PBC;  // Gaussian pairs on integer mantissas
  GaussSum gs[PPT];
  if constexpr (INTEGER) {
#pragma unroll
    for (int h = 0; h < PPT; ++h) {
#pragma unroll
      for (int c = 0; c < 3; ++c) gs[h].f[c] = Acc96{0u, 0u, 0u, ACC_EMPTY};
      gs[h].u = Sum96{0u, 0u, 0u};
      gs[h].bad = 0;
    }
  }
  R fx[PPT] = {}, fy[PPT] = {}, fz[PPT] = {}, u[PPT] = {};
  int nin[PPT] = {};  // Lennard-Jones pairs inside the cutoff (each carries the shift)
  if (pp.pair != BPIMD_PAIR_NONE) {
    for (int base = 0; base < N; base += EXT_CHUNK) {
      const int cnt = min(EXT_CHUNK, N - base);
      __syncthreads();
      for (int q = threadIdx.x; q < cnt; q += EXT_THREADS) {
        const double *r = pos + ((size_t)(base + q) * P + j) * 3;
        R4 t;
        if constexpr (MIXED) { t.x = f32_of_f64(r[0]); t.y = f32_of_f64(r[1]); t.z = f32_of_f64(r[2]); }
        else { t.x = r[0]; t.y = r[1]; t.z = r[2]; }
        if constexpr (MIXED) t.w = 0.0f;
        sr[q] = t;
      }
      __syncthreads();
      if constexpr (INTEGER) {
        if (pp.pair == BPIMD_PAIR_GAUSSIAN) {
#pragma unroll 1
          for (int q = sub; q < cnt; q += SPLIT) {
            const R4 t = sr[q];
#pragma unroll
            for (int h = 0; h < PPT; ++h) {
              const double d[3] = {px[h] - t.x, py[h] - t.y, pz[h] - t.z};
              gauss_pair(d, pp.gm, pp.ge, T63s, gs[h]);
            }
          }
          continue;
        }
      }
      if constexpr (MIXED && !PBC && PPT == 2) {
        if (pp.pair == BPIMD_PAIR_GAUSSIAN) {
          // the two particles in the halves of packed float32 instructions
          const F2 X = pack2(px[0], px[1]), Y = pack2(py[0], py[1]), Z = pack2(pz[0], pz[1]), A = pack2(a, a),
                   K = pack2(1.44269504f, 1.44269504f);
          F2 FX = pack2(fx[0], fx[1]), FY = pack2(fy[0], fy[1]), FZ = pack2(fz[0], fz[1]), U = pack2(u[0], u[1]);
#pragma unroll 4
          for (int q = sub; q < cnt; q += SPLIT) {
            const R4 t = sr[q];
            const F2 dx = add2(X, pack2(-t.x, -t.x)), dy = add2(Y, pack2(-t.y, -t.y)), dz = add2(Z, pack2(-t.z, -t.z));
            const F2 d2 = fma2(dz, dz, fma2(dx, dx, mul2(dy, dy)));  // the rounding of dx dx + dy dy + dz dz
            float e0, e1;
            unpack2(mul2(mul2(A, d2), K), e0, e1);
            const F2 e = pack2(pairg::ex2_approx(e0), pairg::ex2_approx(e1));  // e^(a d2) = 2^(a d2 log2 e)
            FX = fma2(e, dx, FX);
            FY = fma2(e, dy, FY);
            FZ = fma2(e, dz, FZ);
            U = add2(U, e);
          }
          unpack2(FX, fx[0], fx[1]);
          unpack2(FY, fy[0], fy[1]);
          unpack2(FZ, fz[0], fz[1]);
          unpack2(U, u[0], u[1]);
          continue;
        }
      }
      if (pp.pair == BPIMD_PAIR_GAUSSIAN) {
#pragma unroll 4
        for (int q = sub; q < cnt; q += SPLIT) {
          const R4 t = sr[q];
#pragma unroll
          for (int h = 0; h < PPT; ++h) {
            const R dx = img(px[h] - t.x), dy = img(py[h] - t.y), dz = img(pz[h] - t.z);
            const R d2 = dx * dx + dy * dy + dz * dz;
            R e;
            if constexpr (MIXED) e = __expf(a * d2);
            else e = pow2_value(pow2fx::pow2neg_dd((double)d2, pp.g2c, T63s));  // exactly 1 at d = 0
            fx[h] += e * dx; fy[h] += e * dy; fz[h] += e * dz;
            u[h] += e;
          }
        }
      } else {  // Lennard-Jones: force over 24 eps, energy over 4 eps
#pragma unroll 2
        for (int q = sub; q < cnt; q += SPLIT) {
          const R4 t = sr[q];
#pragma unroll
          for (int h = 0; h < PPT; ++h) {
            const R dx = img(px[h] - t.x), dy = img(py[h] - t.y), dz = img(pz[h] - t.z);
            const R r2 = dx * dx + dy * dy + dz * dz;
            if (r2 > (R)0 && r2 < rc2) {
              const R s2 = sig2 / r2, s6 = s2 * s2 * s2;
              const R c = (2 * s6 * s6 - s6) / r2;
              fx[h] += c * dx; fy[h] += c * dy; fz[h] += c * dz;
              u[h] += s6 * s6 - s6;
              ++nin[h];
            }
          }
        }
      }
    }
  }
  double ub[PPT];
#pragma unroll
  for (int h = 0; h < PPT; ++h) {
    if constexpr (INTEGER) {
      if (pp.pair == BPIMD_PAIR_GAUSSIAN) {
        const double nan = __longlong_as_double(0x7ff8000000000000LL);
        fx[h] = gs[h].bad & 1 ? nan : acc_value(gs[h].f[0]);
        fy[h] = gs[h].bad & 2 ? nan : acc_value(gs[h].f[1]);
        fz[h] = gs[h].bad & 4 ? nan : acc_value(gs[h].f[2]);
        u[h] = value96(gs[h].u.lo, gs[h].u.mid, gs[h].u.hi) * 2.168404344971009e-19;  // 2^-62
      }
    }
#pragma unroll
    for (int o = 1; o < SPLIT; o <<= 1) {
      fx[h] += __shfl_xor_sync(0xffffffffu, fx[h], o);
      fy[h] += __shfl_xor_sync(0xffffffffu, fy[h], o);
      fz[h] += __shfl_xor_sync(0xffffffffu, fz[h], o);
      u[h] += __shfl_xor_sync(0xffffffffu, u[h], o);
      nin[h] += __shfl_xor_sync(0xffffffffu, nin[h], o);
    }
    const bool mine = l[h] < N && sub == 0;
    double *f = Fx + ((size_t)l[h] * P + j) * 3;
    if constexpr (MIXED) {
      float ulf = 0.0f;
      if (mine) {
        if (pp.pair == BPIMD_PAIR_GAUSSIAN) u[h] -= 1.0f;  // the self term (d = 0, e = 1) carries no force
        f[0] = f64_of_f32(pp.finv_P * (pp.ffs * fx[h] - pp.fkt * px[h]));
        f[1] = f64_of_f32(pp.finv_P * (pp.ffs * fy[h] - pp.fkt * py[h]));
        f[2] = f64_of_f32(pp.finv_P * (pp.ffs * fz[h] - pp.fkt * pz[h]));
        const float up = pp.pair == BPIMD_PAIR_GAUSSIAN ? pp.fup * u[h] : pp.fup * u[h] - pp.fush * (float)nin[h];
        ulf = pp.finv_P * (up + 0.5f * pp.fkt * (px[h] * px[h] + py[h] * py[h] + pz[h] * pz[h]));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ulf += __shfl_xor_sync(0xffffffffu, ulf, o);
      ub[h] = f64_of_f32(ulf);
    } else {
      double ul = 0.0;
      if (mine) {
        if (pp.pair == BPIMD_PAIR_GAUSSIAN) u[h] -= (R)1;  // the self term (d = 0, e = 1) carries no force
        const double fs = pp.pair == BPIMD_PAIR_GAUSSIAN ? pp.ga * pp.inv_s2 : 24.0 * pp.eps;
        f[0] = pp.inv_P * (fs * (double)fx[h] - pp.kt * rd[h][0]);
        f[1] = pp.inv_P * (fs * (double)fy[h] - pp.kt * rd[h][1]);
        f[2] = pp.inv_P * (fs * (double)fz[h] - pp.kt * rd[h][2]);
        const double up = pp.pair == BPIMD_PAIR_GAUSSIAN ? 0.5 * pp.ga * (double)u[h]
                                                        : 0.5 * (4.0 * pp.eps * (double)u[h] - pp.ushift * nin[h]);
        ul = pp.inv_P * (up + 0.5 * pp.kt * (rd[h][0] * rd[h][0] + rd[h][1] * rd[h][1] + rd[h][2] * rd[h][2]));
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) ul += __shfl_xor_sync(0xffffffffu, ul, o);
      ub[h] = ul;
    }
  }
  // the warps' sums in a fixed order: first halves, then second halves
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int h = 0; h < PPT; ++h) red[h * EXT_WARPS + (threadIdx.x >> 5)] = ub[h];
  }
  __syncthreads();
  double sum = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < PPT * EXT_WARPS; ++q) sum += red[q];
  __syncthreads();
  return sum;
}

// Thermostat kicks of one step, n elements (see md_run): element's amplitude
// c2, or per replica c2r with the packed offsets off.
struct Kicks {
  double *zc;  // null: none wanted
  long long n;
  double c2;
  const double *c2r;
  const long long *off;
  int R;
  uint32_t k0, k1;
  const unsigned long long *step;
  int ahead;   // steps from the counter to the one wanted
};

// The physical force is launched between the recursions and the exterior
// forces and needs only the positions, which were final before the recursions
// could start: it does not wait for them, but runs beside them on the SMs they
// leave free.  Its first block waits for them before it ends, so that the next
// kernel's wait for this one covers both.
__device__ __forceinline__ void after_recursions(bool first_block) {
  pdl_trigger();
  if (first_block) pdl_wait();
}

template <bool MIXED>
__device__ void kicks_block(const Kicks &k, long long blk, long long nblk);

// Block b: the force on bead b / gx of particle block b % gx, then the thermostat
// kicks.  One grid dimension: rows of kicks past the P rows of beads would put
// their sum on y, which ends at 65,535.  Kicks last: as the grid's first columns
// they cost N = 1024, P = 32 (mixed, ten steps) 869 us for 810.
template <bool MIXED, bool PBC>
__global__ void __launch_bounds__(EXT_THREADS) ext_force_kernel(const double *__restrict__ pos,
                                                                double *__restrict__ Fx, int N, int P, PairParams pp,
                                                                double *ubar_part, Kicks kicks, int gx) {
  using R4 = typename std::conditional<MIXED, float4, Dbl3>::type;
  __shared__ R4 sr[EXT_CHUNK];
  __shared__ double red[2 * EXT_WARPS];
  __shared__ unsigned long long T63s[256];  // float64: the table of the integer-pipe power of two
  const int force = gx * P, blk = blockIdx.x;
  if (blk < force) {
    const int j = blk / gx, lb = blk - j * gx;
    const double s = ext_force_body<MIXED, PBC, ext_split(MIXED), ext_ppt(MIXED)>(pos, Fx, N, P, pp, lb, j, sr, red, T63s);
    if (threadIdx.x == 0) ubar_part[blk] = s;
  } else {
    kicks_block<MIXED>(kicks, blk - force, gridDim.x - force);
  }
  after_recursions(blk == 0);
}

// thermostat kicks alone (the cell-list path)
template <bool MIXED>
__global__ void __launch_bounds__(EXT_THREADS) md_kicks_kernel(Kicks kicks) {
  kicks_block<MIXED>(kicks, blockIdx.x, gridDim.x);
}

// ----------------------------------------------------------- replica batches
// Replica r of a batch occupies elements [off[r], off[r] + 3 N_r P_r) of the
// packed arrays; the replica of element e by binary search over off.
__device__ __forceinline__ int replica_of(const long long *__restrict__ off, int R, long long e) {
  int lo = 0, hi = R - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (__ldg(off + mid) <= e) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Blocks blk of nblk of the kicks: four elements a thread.
template <bool MIXED>
__device__ void kicks_block(const Kicks &k, long long blk, long long nblk) {
  if (!k.zc) return;
  const unsigned long long s = *k.step + (unsigned long long)k.ahead;
  for (long long g = blk * (long long)blockDim.x + threadIdx.x; 4 * g < k.n; g += nblk * blockDim.x) {
    double z[4];
    thermostat_kicks<MIXED>(g, s, k.k0, k.k1, z);
    int r = 0;
    long long next = k.n;
    double c2 = k.c2;
    if (k.off) {  // one search a block of four; a replica may end inside it
      r = replica_of(k.off, k.R, 4 * g);
      next = r + 1 < k.R ? __ldg(k.off + r + 1) : k.n;
      c2 = __ldg(k.c2r + r);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const long long e = 4 * g + i;
      while (e >= next && r + 1 < k.R) {
        ++r;
        next = r + 1 < k.R ? __ldg(k.off + r + 1) : k.n;
        c2 = __ldg(k.c2r + r);
      }
      if (e < k.n) k.zc[e] = c2 * z[i];
    }
  }
}

// Trap and pair forces of every replica: entry k of tab is (replica,
// particle block, bead index); the trap frequency and pair parameters are
// shared, 1/P_r is the replica's.  SPLIT lanes per particle, 256 / SPLIT
// particles per block (the batch's pair tile, bpimd_batch_set_pair_tile).
template <bool MIXED, int SPLIT>
__global__ void __launch_bounds__(EXT_THREADS) ext_force_batched(const double *__restrict__ pos,
                                                                 double *__restrict__ Fx,
                                                                 const Workspace *__restrict__ ws,
                                                                 const long long *__restrict__ off,
                                                                 const int4 *__restrict__ tab, int ntab, PairParams pp,
                                                                 double *ubar_part, Kicks kicks, int kick_blocks) {
  using R4 = typename std::conditional<MIXED, float4, Dbl3>::type;
  __shared__ R4 sr[EXT_CHUNK];
  __shared__ double red[2 * EXT_WARPS];
  __shared__ unsigned long long T63s[256];
  if ((int)blockIdx.x < kick_blocks) {
    kicks_block<MIXED>(kicks, blockIdx.x, kick_blocks);
    after_recursions(blockIdx.x == 0);
    return;
  }
  const int b0 = blockIdx.x - kick_blocks, nb = gridDim.x - kick_blocks;
  for (int k = b0; k < ntab; k += nb) {
    const int4 e = tab[k];
    const int N = ws[e.x].N, P = ws[e.x].P;
    PairParams q = pp;
    q.inv_P = ws[e.x].inv_P;
    q.finv_P = f32_of_f64(q.inv_P);
    double s = 0.0;
    if constexpr (MIXED) {
      s = ext_force_body<MIXED, false, SPLIT, 2>(pos + off[e.x], Fx + off[e.x], N, P, q, e.y, e.z, sr, red, T63s);
    } else {  // the tile's halves in turn
#pragma unroll 1
      for (int h = 0; h < 2; ++h)
        s += ext_force_body<MIXED, false, SPLIT, 1>(pos + off[e.x], Fx + off[e.x], N, P, q, 2 * e.y + h, e.z, sr, red, T63s);
    }
    if (threadIdx.x == 0) ubar_part[k] = s;
    __syncthreads();  // sr is reused by the next entry
  }
  after_recursions(blockIdx.x == 0);
}

// energies[4 r + 0..3] of replica r (one block each): V_B, U-bar, kinetic,
// primitive estimator, from the partial sums of the last force pass.
__global__ void __launch_bounds__(MD_THREADS) energies_batched(const Workspace *__restrict__ ws,
                                                               const double *__restrict__ VBr,
                                                               const double *__restrict__ ubar_part,
                                                               const int *__restrict__ ext_first,
                                                               const double *__restrict__ spring_part,
                                                               const int *__restrict__ blk_first, int ntab,
                                                               double half_m, double *energies) {
  __shared__ double red[MD_THREADS / 32];
  const int r = blockIdx.x;
  const Workspace &w = ws[r];
  double sp = 0.0, ub = 0.0, ke = 0.0;
  for (int q = blk_first[r] + threadIdx.x; q < blk_first[r + 1]; q += blockDim.x) {
    sp += spring_part[q];
    ke += spring_part[ntab + q];
  }
  for (int q = ext_first[r] + threadIdx.x; q < ext_first[r + 1]; q += blockDim.x) ub += ubar_part[q];
  sp = block_sum(sp, red);
  ub = block_sum(ub, red);
  ke = block_sum(ke, red);
  if (threadIdx.x == 0) {
    double *en = energies + 4 * (size_t)r;
    en[0] = VBr[r];
    en[1] = ub;
    en[2] = half_m * ke;
    en[3] = 1.5 * (double)w.N * (double)w.P / w.beta - sp + ub;
    for (int i = 0; i < 4; ++i)
      if (!isfinite(en[i])) atomicOr(w.status, ST_NONFINITE);
  }
}

__global__ void __launch_bounds__(MD_THREADS) ke_kernel(const double *__restrict__ v, long long n, double half_m,
                                                        double *ke_part) {
  __shared__ double red[MD_THREADS / 32];
  double acc = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n; e += (long long)gridDim.x * blockDim.x)
    acc += v[e] * v[e];
  const double s = block_sum(acc, red);
  if (threadIdx.x == 0) ke_part[blockIdx.x] = half_m * s;
}

// energies[0..3] = V_B, U-bar, kinetic, primitive estimator 3NP/(2 beta) - <springs> + U-bar,
// with <springs> = sum_l E_int + sum Pr[l -> u<=l] (1/2)k d^2 + sum Pr[l -> l+1] link_l.
__global__ void __launch_bounds__(ENERGY_THREADS) energies_kernel(Workspace w, const double *VB, const double *ubar_part,
                                                              int n_ubar, const double *ke_part, int n_ke,
                                                              const double *spring_part, double *energies) {
  __shared__ double red[ENERGY_THREADS / 32];
  double sp = 0.0, ub = 0.0, ke = 0.0;
  for (int q = threadIdx.x; q < w.NB; q += blockDim.x) sp += spring_part[q];
  for (int q = threadIdx.x; q < n_ubar; q += blockDim.x) ub += ubar_part[q];
  for (int q = threadIdx.x; q < n_ke; q += blockDim.x) ke += ke_part[q];
  sp = block_sum(sp, red);
  ub = block_sum(ub, red);
  ke = block_sum(ke, red);
  if (threadIdx.x == 0) {
    energies[0] = *VB;
    energies[1] = ub;
    energies[2] = ke;
    energies[3] = 1.5 * (double)w.N * (double)w.P / w.beta - sp + ub;
    for (int i = 0; i < 4; ++i)
      if (!isfinite(energies[i])) atomicOr(w.status, ST_NONFINITE);
  }
}

struct MDParams {
  long long n;
  double half_dt_over_m, half_dt, c1, c2;
  PairParams pp;
  int cell_nc;  // > 0: Lennard-Jones by cell lists with cell_nc^3 cells per bead index
  uint32_t k0, k1;
};

int md_params(const bpimd_config &c, MDParams &p) {
  if (!(c.dt > 0.0) || !std::isfinite(c.dt) || !(c.gamma >= 0.0) || !std::isfinite(c.gamma)) return BPIMD_ERR_ARG;
  if (!(c.kT_bead >= 0.0) || !std::isfinite(c.kT_bead) || !(c.omega0 >= 0.0) || !std::isfinite(c.omega0))
    return BPIMD_ERR_ARG;
  if (c.pair_type != BPIMD_PAIR_NONE && c.pair_type != BPIMD_PAIR_GAUSSIAN && c.pair_type != BPIMD_PAIR_LJ)
    return BPIMD_ERR_ARG;
  if (c.pair_type != BPIMD_PAIR_NONE &&
      (!std::isfinite(c.pair_a) || !(c.pair_b > 0.0) || !std::isfinite(c.pair_b)))
    return BPIMD_ERR_ARG;
  const double L = c.box_L;
  if (c.pair_type == BPIMD_PAIR_LJ) {
    // a cutoff is required; in a box it may not exceed half the side (minimum image)
    if (!(c.pair_rc > 0.0) || !std::isfinite(c.pair_rc)) return BPIMD_ERR_ARG;
    if (L > 0.0 && c.pair_rc > 0.5 * L) return BPIMD_ERR_ARG;
  }
  const double kT = c.kT_bead > 0.0 ? c.kT_bead : 1.0 / c.beta;
  p.n = (long long)c.N * c.P * 3;
  p.half_dt_over_m = 0.5 * c.dt / c.m;
  p.half_dt = 0.5 * c.dt;
  p.c1 = std::exp(-c.gamma * c.dt);
  p.c2 = std::sqrt((1.0 - p.c1 * p.c1) * kT / c.m);
  PairParams &q = p.pp;
  q = PairParams{};
  q.pair = c.pair_type;
  q.inv_P = 1.0 / c.P;
  q.kt = c.m * c.omega0 * c.omega0;
  if (c.pair_type == BPIMD_PAIR_GAUSSIAN) {
    q.ga = c.pair_a;
    q.inv_s2 = 1.0 / (c.pair_b * c.pair_b);
    q.g2c = 0.5 * q.inv_s2 * 1.4426950408889634;  // log2(e) / (2 s^2)
    // g2c = gm 2^(ge - 63); where 1/s^2 has left the float64 range e is 0 or 1
    int ex = 0;
    const double m = std::frexp(q.g2c, &ex);  // m in [0.5, 1)
    const bool normal = std::isfinite(q.g2c) && q.g2c >= 2.3e-308;
    q.gm = normal ? (unsigned long long)std::ldexp(m, 64) : 1ull << 63;
    q.ge = normal ? ex - 1 : (q.g2c < 1.0 ? -1100 : 1100);
  }
  if (c.pair_type == BPIMD_PAIR_LJ) {
    q.eps = c.pair_a;
    q.sig2 = c.pair_b * c.pair_b;
    q.rc2 = c.pair_rc * c.pair_rc;
    const double sr2 = q.sig2 / q.rc2, sr6 = sr2 * sr2 * sr2;
    q.ushift = 4.0 * c.pair_a * (sr6 * sr6 - sr6);
  }
  q.L = L > 0.0 ? L : 0.0;
  q.invL = L > 0.0 ? 1.0 / L : 0.0;
  q.Lscale = (float)(q.L / 4294967296.0);
  q.pbc = L > 0.0 ? 1 : 0;
  q.fa = (float)(-0.5 * q.inv_s2);
  q.ffs = (float)(c.pair_type == BPIMD_PAIR_GAUSSIAN ? q.ga * q.inv_s2 : 24.0 * q.eps);
  q.fup = (float)(c.pair_type == BPIMD_PAIR_GAUSSIAN ? 0.5 * q.ga : 2.0 * q.eps);
  q.fkt = (float)q.kt;
  q.fL = (float)q.L;
  q.finvL = (float)q.invL;
  q.fsig2 = (float)q.sig2;
  q.frc2 = (float)q.rc2;
  q.fush = (float)(0.5 * q.ushift);
  q.finv_P = (float)q.inv_P;
  p.cell_nc = 0;
  if (c.pair_type == BPIMD_PAIR_LJ && L > 0.0) {
    const int nc = (int)std::floor(L / c.pair_rc);
    if (nc >= 3 && (long long)nc * nc * nc * c.P <= (1LL << 26)) p.cell_nc = nc;
  }
  p.k0 = (uint32_t)c.seed;
  p.k1 = (uint32_t)(c.seed >> 32);
  return BPIMD_OK;
}

int grid_for(long long work, int threads) {
  const long long b = (work + threads - 1) / threads;
  const long long cap = (long long)sm_count() * 8;
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

// Which thermostat kicks a force pass forms beside it: those of the step the
// counter shows, of the one after it, or none.
enum KickStep { KICKS_NOW = 0, KICKS_NEXT = 1, KICKS_NONE = -1 };

Kicks kicks_of(const MDState &md, const MDParams &p, KickStep ks) {
  Kicks k = {};
  k.zc = (ks == KICKS_NONE || p.c1 == 1.0) ? nullptr : md.zc;  // no friction: no kicks
  k.n = p.n;
  k.c2 = p.c2;
  k.c2r = md.c2r;
  k.k0 = p.k0;
  k.k1 = p.k1;
  k.step = md.step;
  k.ahead = ks == KICKS_NEXT ? 1 : 0;
  return k;
}

// md.F = exchange force (Algorithm 1) and md.Fx = physical force of pos, with
// the U-bar partials and the thermostat kicks of step `ks`.
int total_force(bpimd_ctx *ctx, const MDParams &p, const double *pos, KickStep ks) {
  MDState &md = ctx->md;
  cudaStream_t s = ctx->stream;
  const Kicks kicks = kicks_of(md, p, ks);
  const int kick_blocks = kicks.zc ? grid_for((p.n + 3) / 4, EXT_THREADS) : 0;
  if (p.cell_nc > 0) {
    // the cell-list kernels run beside the whole evaluation, on a stream of their own
    if (cudaEventRecord(md.fork, s) != cudaSuccess || cudaStreamWaitEvent(md.side, md.fork, 0) != cudaSuccess)
      return BPIMD_ERR_CUDA;
    if (kicks.zc) {
      if (ctx->w.bead32) md_kicks_kernel<true><<<kick_blocks, EXT_THREADS, 0, md.side>>>(kicks);
      else md_kicks_kernel<false><<<kick_blocks, EXT_THREADS, 0, md.side>>>(kicks);
    }
    int rc = cell_list_forces(pos, md.Fx, ctx->cfg.N, ctx->cfg.P, p.pp, ctx->w.bead32, md.cells, md.ubar_part,
                              md.side) == cudaSuccess ? BPIMD_OK : BPIMD_ERR_CUDA;
    if (cudaEventRecord(md.join, md.side) != cudaSuccess) rc = BPIMD_ERR_CUDA;
    const int re = evaluate(ctx, pos, md.VB, md.F);
    if (cudaStreamWaitEvent(s, md.join, 0) != cudaSuccess) return BPIMD_ERR_CUDA;
    return rc != BPIMD_OK ? rc : re;
  }
  const int N = ctx->cfg.N, P = ctx->cfg.P, pb = ext_particles(ctx->w.bead32), gx = (N + pb - 1) / pb;
  if (P > 65535) return BPIMD_ERR_CUDA;  // as ever: a row of the grid a bead
  const int grid = gx * P + kick_blocks;
  return evaluate(ctx, pos, md.VB, md.F, [&] {
    auto go = [&](auto kernel) {
      return launch_pdl(kernel, grid, EXT_THREADS, 0, s, pos, md.Fx, N, P, p.pp, md.ubar_part, kicks, gx);
    };
    if (ctx->w.bead32) return p.pp.pbc ? go(ext_force_kernel<true, true>) : go(ext_force_kernel<true, false>);
    return p.pp.pbc ? go(ext_force_kernel<false, true>) : go(ext_force_kernel<false, false>);
  });
}

// Closing B of a step (K) and B A O A of the next (A), in one pass over the
// arrays where both are due.
template <bool K, bool A>
int launch_update(bpimd_ctx *ctx, const MDParams &p, double *pos, double *vel) {
  MDState &md = ctx->md;
  return launch_pdl(md_update_kernel<K, A>, grid_for((p.n + 1) / 2, MD_THREADS), MD_THREADS, 0, ctx->stream, pos, vel,
                    md.F, md.Fx, p.c1 == 1.0 ? nullptr : md.zc, p.n, p.half_dt_over_m, p.half_dt, p.c1, md.step) ==
                 cudaSuccess
             ? BPIMD_OK
             : BPIMD_ERR_CUDA;
}

// Steps of one call: `force(ks)` enqueues a force pass.  The first B A O A, then
// nsteps - 1 times a force pass with the closing B and the next step's B A O A
// (captured once into a graph bound to the buffers, not on the legacy default
// stream), then the last force pass and closing B.
template <typename Force>
int run_steps(bpimd_ctx *ctx, const MDParams &p, double *pos, double *vel, int32_t nsteps, Force force) {
  MDState &md = ctx->md;
  int rc = force(nsteps > 0 ? KICKS_NOW : KICKS_NONE);  // the caller may have moved the positions since the last call
  if (rc != BPIMD_OK || nsteps == 0) return rc;
  if ((rc = launch_update<false, true>(ctx, p, pos, vel)) != BPIMD_OK) return rc;
  auto step = [&] {
    const int r = force(KICKS_NEXT);
    return r != BPIMD_OK ? r : launch_update<true, true>(ctx, p, pos, vel);
  };
  const bool use_graph = ctx->stream != nullptr && nsteps > 1;
  if (use_graph && (!md.exec || md.g_pos != pos || md.g_vel != vel)) {
    if (md.exec) { cudaGraphExecDestroy(md.exec); md.exec = nullptr; }
    if (md.graph) { cudaGraphDestroy(md.graph); md.graph = nullptr; }
    if (cudaStreamBeginCapture(ctx->stream, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return BPIMD_ERR_CUDA;
    const int rc_step = step();
    const cudaError_t e = cudaStreamEndCapture(ctx->stream, &md.graph);
    if (rc_step != BPIMD_OK || e != cudaSuccess || cudaGraphInstantiate(&md.exec, md.graph, 0) != cudaSuccess) {
      cudaGetLastError();
      return BPIMD_ERR_CUDA;
    }
    md.g_pos = pos;
    md.g_vel = vel;
  }
  for (int32_t k = 1; k < nsteps && rc == BPIMD_OK; ++k) {
    if (use_graph) rc = cudaGraphLaunch(md.exec, ctx->stream) == cudaSuccess ? BPIMD_OK : BPIMD_ERR_CUDA;
    else rc = step();
  }
  if (rc == BPIMD_OK) rc = force(KICKS_NONE);
  if (rc == BPIMD_OK) rc = launch_update<true, false>(ctx, p, pos, vel);
  if (rc == BPIMD_OK) md.steps_taken += (uint64_t)nsteps;
  return rc;
}

int md_alloc(bpimd_ctx *ctx, const MDParams &p) {
  MDState &md = ctx->md;
  if (p.cell_nc > 0) {
    const size_t bytes = cell_list_bytes(ctx->cfg.N, ctx->cfg.P, p.cell_nc, ctx->w.bead32);
    if (cudaMalloc(&md.cell_block, bytes) != cudaSuccess) {
      cudaGetLastError();
      return BPIMD_ERR_NOMEM;
    }
    cell_list_layout(md.cells, (char *)md.cell_block, ctx->cfg.N, ctx->cfg.P, p.cell_nc, ctx->w.bead32);
    if (cudaStreamCreateWithFlags(&md.side, cudaStreamNonBlocking) != cudaSuccess ||
        cudaEventCreateWithFlags(&md.fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&md.join, cudaEventDisableTiming) != cudaSuccess) {
      cudaGetLastError();
      md_free(&md);
      return BPIMD_ERR_NOMEM;
    }
  }
  const size_t n = (size_t)ctx->cfg.N * ctx->cfg.P * 3;
  md.ext_blocks = p.cell_nc > 0 ? cell_list_partials(ctx->cfg.N, ctx->cfg.P)
                                 : ((ctx->cfg.N + ext_particles(ctx->w.bead32) - 1) / ext_particles(ctx->w.bead32)) * ctx->cfg.P;
  md.ke_blocks = grid_for((long long)n, MD_THREADS);
  md.spring_blocks = ctx->w.NB;
  if (cudaMalloc(&md.F, sizeof(double) * n) != cudaSuccess || cudaMalloc(&md.Fx, sizeof(double) * n) != cudaSuccess ||
      cudaMalloc(&md.zc, sizeof(double) * n) != cudaSuccess || cudaMalloc(&md.VB, sizeof(double)) != cudaSuccess ||
      cudaMalloc(&md.ubar_part, sizeof(double) * md.ext_blocks) != cudaSuccess ||
      cudaMalloc(&md.ke_part, sizeof(double) * md.ke_blocks) != cudaSuccess ||
      cudaMalloc(&md.spring_part, sizeof(double) * md.spring_blocks) != cudaSuccess ||
      cudaMalloc(&md.step, sizeof(unsigned long long)) != cudaSuccess) {
    cudaGetLastError();
    md_free(&md);
    return BPIMD_ERR_NOMEM;
  }
  if (cudaMemsetAsync(md.step, 0, sizeof(unsigned long long), ctx->stream) != cudaSuccess) return BPIMD_ERR_CUDA;
  md.ready = true;
  return BPIMD_OK;
}

}  // namespace

void md_init(MDState *md) { *md = MDState{}; }

void md_free(MDState *md) {
  cudaFree(md->VBr);
  cudaFree(md->c2r);
  cudaFree(md->ext_tab);
  cudaFree(md->ext_first);
  cudaFree(md->blk_first);
  if (md->exec) cudaGraphExecDestroy(md->exec);
  if (md->graph) cudaGraphDestroy(md->graph);
  cudaFree(md->F);
  cudaFree(md->Fx);
  cudaFree(md->zc);
  if (md->side) cudaStreamDestroy(md->side);
  if (md->fork) cudaEventDestroy(md->fork);
  if (md->join) cudaEventDestroy(md->join);
  cudaFree(md->VB);
  cudaFree(md->ubar_part);
  cudaFree(md->ke_part);
  cudaFree(md->spring_part);
  cudaFree(md->step);
  cudaFree(md->cell_block);
  *md = MDState{};
}

int md_run(bpimd_ctx *ctx, double *pos, double *vel, int32_t nsteps, double *energies) {
  MDParams p;
  int rc = md_params(ctx->cfg, p);
  if (rc != BPIMD_OK) return rc;
  MDState &md = ctx->md;
  if (!md.ready && (rc = md_alloc(ctx, p)) != BPIMD_OK) return rc;
  // stage profiling is not recorded inside MD steps
  const bool prof = ctx->prof_on;
  ctx->prof_on = false;
  rc = run_steps(ctx, p, pos, vel, nsteps, [&](KickStep ks) { return total_force(ctx, p, pos, ks); });
  if (rc == BPIMD_OK && energies) {
    cudaStream_t s = ctx->stream;
    const int g1 = md.ke_blocks;
    ke_kernel<<<g1, MD_THREADS, 0, s>>>(vel, p.n, 0.5 * ctx->cfg.m, md.ke_part);
    if (cudaGetLastError() != cudaSuccess || launch_spring_expectation(ctx->w, md.spring_part, s) != cudaSuccess)
      rc = BPIMD_ERR_CUDA;
    if (rc == BPIMD_OK) {
      energies_kernel<<<1, ENERGY_THREADS, 0, s>>>(ctx->w, md.VB, md.ubar_part, md.ext_blocks, md.ke_part, g1,
                                              md.spring_part, energies);
      if (cudaGetLastError() != cudaSuccess) rc = BPIMD_ERR_CUDA;
    }
  }
  ctx->prof_on = prof;
  return rc;
}

// ----------------------------------------------------------- replica batches
// bpimd_step on a batch context: every replica advances by the same BAOAB
// steps (shared dt, gamma, trap, Gaussian pair potential and seed; each
// replica thermostatted at its own kT = 1/beta_r unless cfg.kT_bead > 0).
// The steps run as a single system's (run_steps), with the batch evaluation and
// the batched trap and pair forces.  Thermostat noise: Philox4x32-10 with the
// element index of the packed arrays as the counter.
namespace {

// (replica, particle block, bead index) table of the batched pair forces for
// `lanes` lanes per particle (256 / lanes particles per block)
void pair_table(const bpimd_ctx *ctx, int lanes, std::vector<int4> &tab, std::vector<int> &ext_first) {
  const int R = ctx->R, pb = 2 * EXT_THREADS / lanes;
  tab.clear();
  ext_first.assign(R + 1, 0);
  for (int r = 0; r < R; ++r) {
    const Workspace &w = ctx->h_ws[r];
    ext_first[r] = (int)tab.size();
    for (int j = 0; j < w.P; ++j)
      for (int lb = 0; lb * pb < w.N; ++lb) tab.push_back(make_int4(r, lb, j, 0));
  }
  ext_first[R] = (int)tab.size();
}

int md_alloc_batched(bpimd_ctx *ctx, const MDParams &p) {
  MDState &md = ctx->md;
  const int R = ctx->R;
  const size_t n = (size_t)ctx->total_elems;
  std::vector<int4> tab;
  std::vector<int> ext_first, blk_first(R + 1);
  pair_table(ctx, 8, tab, ext_first);  // the largest table: its size is the capacity
  md.ext_cap = (int)tab.size();
  pair_table(ctx, ctx->pair_lanes, tab, ext_first);
  int blk = 0;
  for (int r = 0; r < R; ++r) {
    blk_first[r] = blk;
    blk += ctx->h_ws[r].NB;
  }
  blk_first[R] = blk;
  md.n_ext = (int)tab.size();
  md.spring_blocks = 2 * ctx->n_blk_tab;  // spring and kinetic parts
  md.ke_blocks = 0;
  md.ext_blocks = md.n_ext;
  std::vector<double> c2(R);
  for (int r = 0; r < R; ++r) {
    const double kT = ctx->cfg.kT_bead > 0.0 ? ctx->cfg.kT_bead : 1.0 / ctx->h_ws[r].beta;
    c2[r] = std::sqrt((1.0 - p.c1 * p.c1) * kT / ctx->cfg.m);
  }
  if (cudaMalloc(&md.F, sizeof(double) * n) != cudaSuccess || cudaMalloc(&md.Fx, sizeof(double) * n) != cudaSuccess ||
      cudaMalloc(&md.zc, sizeof(double) * n) != cudaSuccess || cudaMalloc(&md.VBr, sizeof(double) * R) != cudaSuccess ||
      cudaMalloc(&md.c2r, sizeof(double) * R) != cudaSuccess ||
      cudaMalloc(&md.ext_tab, sizeof(int4) * md.ext_cap) != cudaSuccess ||
      cudaMalloc(&md.ext_first, sizeof(int) * (R + 1)) != cudaSuccess ||
      cudaMalloc(&md.blk_first, sizeof(int) * (R + 1)) != cudaSuccess ||
      cudaMalloc(&md.ubar_part, sizeof(double) * md.ext_cap) != cudaSuccess ||
      cudaMalloc(&md.spring_part, sizeof(double) * md.spring_blocks) != cudaSuccess ||
      cudaMalloc(&md.step, sizeof(unsigned long long)) != cudaSuccess) {
    cudaGetLastError();
    md_free(&md);
    return BPIMD_ERR_NOMEM;
  }
  cudaStream_t s = ctx->stream;
  if (cudaMemcpyAsync(md.c2r, c2.data(), sizeof(double) * R, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(md.ext_tab, tab.data(), sizeof(int4) * md.n_ext, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(md.ext_first, ext_first.data(), sizeof(int) * (R + 1), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaMemcpyAsync(md.blk_first, blk_first.data(), sizeof(int) * (R + 1), cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaMemsetAsync(md.step, 0, sizeof(unsigned long long), s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)  // the host tables go out of scope
    return BPIMD_ERR_CUDA;
  md.ready = true;
  return BPIMD_OK;
}

int total_force_batched(bpimd_ctx *ctx, const MDParams &p, const double *pos, KickStep ks) {
  MDState &md = ctx->md;
  Kicks kicks = kicks_of(md, p, ks);
  kicks.off = ctx->d_off;
  kicks.R = ctx->R;
  const int kick_blocks = kicks.zc ? grid_for((p.n + 3) / 4, EXT_THREADS) : 0;
  const int grid = kick_blocks + (md.n_ext < sm_count() * 12 ? md.n_ext : sm_count() * 12);
  return evaluate_batched(ctx, pos, md.VBr, md.F, [&] {
    auto go = [&](auto kernel) {
      return launch_pdl(kernel, grid, EXT_THREADS, 0, ctx->stream, pos, md.Fx, ctx->d_ws, ctx->d_off, md.ext_tab,
                        md.n_ext, p.pp, md.ubar_part, kicks, kick_blocks);
    };
    const bool m = ctx->w.bead32;
    switch (ctx->pair_lanes) {
      case 2: return m ? go(ext_force_batched<true, 2>) : go(ext_force_batched<false, 2>);
      case 8: return m ? go(ext_force_batched<true, 8>) : go(ext_force_batched<false, 8>);
      default: return m ? go(ext_force_batched<true, 4>) : go(ext_force_batched<false, 4>);
    }
  });
}

}  // namespace

// A new pair tile for a batch: with MD state allocated, rebuild the pair-force
// table (within the capacity of the 8-lane table) and drop the captured step,
// which is recaptured by the next bpimd_step; forces, velocities and the
// thermostat counter are kept, so a trajectory goes on unchanged.
int md_set_pair_tile(bpimd_ctx *ctx, int lanes) {
  MDState &md = ctx->md;
  if (md.ready && lanes != ctx->pair_lanes) {
    std::vector<int4> tab;
    std::vector<int> ext_first;
    pair_table(ctx, lanes, tab, ext_first);
    if ((int)tab.size() > md.ext_cap) return BPIMD_ERR_STATE;
    cudaStream_t s = ctx->stream;
    if (cudaStreamSynchronize(s) != cudaSuccess ||
        cudaMemcpyAsync(md.ext_tab, tab.data(), sizeof(int4) * tab.size(), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaMemcpyAsync(md.ext_first, ext_first.data(), sizeof(int) * ext_first.size(), cudaMemcpyHostToDevice, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)  // the host tables go out of scope
      return BPIMD_ERR_CUDA;
    md.n_ext = (int)tab.size();
    md.ext_blocks = md.n_ext;
    if (md.exec) { cudaGraphExecDestroy(md.exec); md.exec = nullptr; }
    if (md.graph) { cudaGraphDestroy(md.graph); md.graph = nullptr; }
    md.g_pos = md.g_vel = nullptr;
  }
  ctx->pair_lanes = lanes;
  return BPIMD_OK;
}

int md_run_batched(bpimd_ctx *ctx, double *pos, double *vel, int32_t nsteps, double *energies) {
  bpimd_config c = ctx->cfg;
  if (c.pair_type == BPIMD_PAIR_LJ) return BPIMD_ERR_ARG;  // batches have no periodic box
  c.N = 1;
  c.P = 2;
  c.beta = 1.0;  // md_params' kT only fills p.c2, which batches replace per replica
  MDParams p;
  int rc = md_params(c, p);
  if (rc != BPIMD_OK) return rc;
  p.n = ctx->total_elems;
  MDState &md = ctx->md;
  if (!md.ready && (rc = md_alloc_batched(ctx, p)) != BPIMD_OK) return rc;
  const bool prof = ctx->prof_on;
  ctx->prof_on = false;
  rc = run_steps(ctx, p, pos, vel, nsteps, [&](KickStep ks) { return total_force_batched(ctx, p, pos, ks); });
  if (rc == BPIMD_OK && energies) {
    cudaStream_t s = ctx->stream;
    if (launch_spring_expectation_batched(ctx->d_ws, ctx->d_blk_tab, ctx->n_blk_tab, ctx->d_off, vel, md.spring_part,
                                          s) != cudaSuccess)
      rc = BPIMD_ERR_CUDA;
    if (rc == BPIMD_OK) {
      energies_batched<<<ctx->R, MD_THREADS, 0, s>>>(ctx->d_ws, md.VBr, md.ubar_part, md.ext_first, md.spring_part,
                                                     md.blk_first, ctx->n_blk_tab, 0.5 * ctx->cfg.m, energies);
      if (cudaGetLastError() != cudaSuccess) rc = BPIMD_ERR_CUDA;
    }
  }
  ctx->prof_on = prof;
  return rc;
}

}  // namespace bpimd
