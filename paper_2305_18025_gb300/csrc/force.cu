// Connection probabilities fused with the exterior-bead forces.
//
//   Pr[l -> u] (u <= l) = y_{u-1} g(u,l) mu_l / (N y_N)     (Eq. close-cycle-probability)
//   Pr[l -> l+1]        = 1 - y_l B_{l+1} / (N y_N)          (Eq. direct-link-probability)
//   Pr[l -> u]          = 0 for u > l+1                      (Lemma zero-connection-probability)
// The N x N matrix is never stored: the pass goes by tiles of 32 particles and
// forms (Eq. force-on-1-sum-neighbors, Eq. force-on-P-sum-neighbors)
//   F_l^P = -m w_P^2 [ (sum_u Pr[l->u]) (r_l^P - r_l^{P-1}) + sum_u Pr[l->u] (r_l^P - r_u^1) ]
//   F_l^1 = -m w_P^2 [ (sum_l' Pr[l'->l]) (r_l^1 - r_l^2) + sum_l' Pr[l'->l] (r_l^1 - r_l'^P) ]
// i.e. the per-neighbour sums of the paper distributed over their terms.
// Precision forms: bead differences in float64 (FP64) or float32 (mixed
// forms, from the high/low parts or the fixed-point copies); products and sums
// on 64-bit integer mantissas (FP64) or as float32 pairs (mixed forms); the direct
// links and the results in float64.
#include <type_traits>

#include "bpimd_internal.cuh"
#include "pairg.cuh"

namespace bpimd {
namespace {

// (float32 estimate of the triangular root, corrected with integer tests:
// no float64 instruction)
__device__ __forceinline__ void block_coords_f(int blk, int &t, int &s) {
  int tt = (int)((sqrtf(8.0f * (float)blk + 1.0f) - 1.0f) * 0.5f);
  while ((tt + 1) * (tt + 2) / 2 <= blk) ++tt;
  while (tt * (tt + 1) / 2 > blk) --tt;
  t = tt;
  s = blk - tt * (tt + 1) / 2;
}

__device__ __forceinline__ xd alpha_of(const Workspace &w, int a) {  // y_a / (N y_N)
  return xmul(xd{w.yfm[a], w.yfe[a]}, xd{w.scal[1], w.scal_i[0]});
}
__device__ __forceinline__ xd mu_of(const Workspace &w, int b) {
  const int r = w.N - 1 - b;  // backward row index of mu_b (0-based mu~_b = Yb[N-1-b])
  return xd{w.ybm[r], w.ybe[r]};
}

// 2^e as a double for e in the normal range (0 below it), built from the bits.
__device__ __forceinline__ double pow2_normal(int e) {
  return e < -1022 ? 0.0 : __longlong_as_double((long long)(min(e, 1023) + 1023) << 52);
}

// Pr[p -> p+1] = 1 - y_{p+1} B_{p+2} / (N y_N) (0-based p; Eq.
// direct-link-probability) with B_{p+2} = Yb[N-p-1] / c_{p+1}: one mantissa
// product and quotient in float64, the exponents summed as integers.
__device__ __forceinline__ double direct_link_fast(const Workspace &w, int p) {
  const double ym = w.yfm[p + 1], bm = w.ybm[w.N - p - 1], cm = w.ccm[p], zm = w.scal[1];
  const int e = w.yfe[p + 1] + w.ybe[w.N - p - 1] - w.cce[p] + w.scal_i[0];
  return 1.0 - ((ym * bm) * zm / cm) * pow2_normal(e);
}

template <bool PBC>
__device__ __forceinline__ double img(const Workspace &w, double d) {
  return PBC ? d - w.L * rint(d * w.invL) : d;
}

// ------------------------------------------- exterior forces by whole tiles
// Item 2k is row tile NT-1-k (bead P of its 32 particles b, against every
// source a <= b), item 2k+1 column tile k (bead 1 of its 32 particles a,
// against every b >= a): decreasing sizes.  A lane owns one particle; the
// partners are dealt out in chunks over the item's cluster (CL CTAs) and
// staged in shared memory, a warp taking an eighth of a chunk.  With mu_b and
// 1/(N y_N) taken out of a row's sum, and y_a and 1/(N y_N) out of a column's,
//   row b    : mu_b / (N y_N) sum_a y_a g(a,b) (r_b^P - r_a^1)
//   column a : y_a / (N y_N) sum_b mu_b g(a,b) (r_b^P - r_a^1)
// a pair is one product and three products with the difference's components.
//   Mixed forms: unevaluated float32 pairs (products by FMA, sums by TwoSum:
//   2^-46 relative) on the float32 pipe; the powers of two of all factors,
//   the taken-out ones included, scale the pair, so a term is at most 2.  High
//   parts are the nearest float32: a weight's error over random mantissas is then
//   0.12 2^-46 (rms; 0.91 at most, 0.00 on average), where high parts cut off gave
//   0.89 (3.1, -0.80) and one cut of the 64-bit product 0.42 (1.0, -0.36) at 4-12 %
//   of the pass (N = 1024, P = 32: 56.6 us for 55.6; 152 replicas of 1024: 784 us
//   for 701).
//   FP64: 64-bit integer mantissas, signed 64-bit sums with a running exponent
//   a lane and component (2^-57 of the largest term of a group of four); GB300's
//   float64 pipe retires ~1.7 lanes a clock, so it forms the differences only.
// The sums of the probabilities themselves are not needed: by the recursions'
// own equations sum_u Pr[l->u] + Pr[l->l+1] = 1, and so for the columns.
// Partial sums meet in shared memory, then in the cluster's first CTA, in a
// fixed order: nothing O(N^2) is written, and there are no atomics.
// Each pair is formed twice (row and column), which costs less than the
// transposed reduction, the global partial sums, the fence and the counters
// of a pass that forms it once.
struct PSum {  // FP64: v 2^(E - 61)
  long long v;
  int E;
};

__device__ __forceinline__ unsigned long long mant64(double m) {  // [1, 2) -> [2^63, 2^64)
  return ((unsigned long long)__double_as_longlong(m) << 11) | (1ull << 63);
}

// |x| as a mantissa in [2^62, 2^63) (value M 2^(e - 62)) times the term t:
// the high product, its exponent e, its sign; a zero has the exponent NO_TERM
constexpr int NO_TERM = -(1 << 30);
__device__ __forceinline__ unsigned long long diff_term(unsigned long long t, double x, int &e, int &sgn, bool &bad) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int hi = (int)(b >> 32), ex = (hi >> 20) & 0x7ff;
  sgn = hi >> 31;
  e = ex ? ex - 1023 : NO_TERM;
  bad = ex == 0x7ff;
  return pow2fx::mulhi(t, ((b << 10) & 0x3FFFFFFFFFFFFFFFull) | (1ull << 62));
}

// stores into the cluster's first CTA, and the cluster barrier
__device__ __forceinline__ unsigned first_cta(const void *p) {
  unsigned r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"((unsigned)__cvta_generic_to_shared(p)));
  return r;
}
__device__ __forceinline__ void cluster_store(const void *p, long long v) {
  asm volatile("st.shared::cluster.b64 [%0], %1;" ::"r"(first_cta(p)), "l"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(const void *p, int v) {
  asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(first_cta(p)), "r"(v) : "memory");
}
__device__ __forceinline__ void cluster_store(const void *p, float v) { cluster_store(p, __float_as_int(v)); }
__device__ __forceinline__ void cluster_arrive_release() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait_acquire() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ long long shift_in(long long v, int k) { return v >> min(k, 63); }

// a + b, |b| < 2^62; |a| stays below 2^62
__device__ __forceinline__ void psum_add(PSum &a, const PSum &b) {
  const int E = max(a.E, b.E);
  a.v = shift_in(a.v, E - a.E) + shift_in(b.v, E - b.E);
  const int h = (int)(a.v >> 32), big = (h ^ (h >> 31)) >> 30;  // 0 or 1
  a.v >>= big;
  a.E = E + big;
}

// Mixed forms: s + c with every rounding error of s in c
__device__ __forceinline__ void two_sum(float &s, float &c, float x) {
  const float t = s + x, bp = t - s;
  c += (s - (t - bp)) + (x - bp);
  s = t;
}
// a mantissa in [1, 2) as the nearest float32 and the rest (to 2^-49)
__device__ __forceinline__ void mant_hl(double m, float &h, float &l) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(m);
  h = __uint_as_float(0x3F800000u + (((unsigned)(b >> 29) & 0x7FFFFFu) + ((unsigned)(b >> 28) & 1u)));
  l = (float)((int)((unsigned)b << 3) >> 3) * 2.2204460492503131e-16f;  // 2^-52
}
__device__ __forceinline__ void mant_hl(float m, float &h, float &l) {
  h = m;
  l = 0.0f;
}

constexpr int PROB_THREADS = 256, PROB_WARPS = PROB_THREADS / 32;
constexpr int PROB_MAX_CL = 8;
constexpr int PROB_CHUNK = 256;  // most partners staged at a time

// Sums of a warp or a CTA: mixed forms (s, c) per component, FP64 v, E and the
// non-finite flag.
template <bool F64>
struct SumSlot;
template <>
struct SumSlot<false> {
  float s[3][TILE], c[3][TILE];
};
template <>
struct SumSlot<true> {
  long long v[3][TILE];
  int E[3][TILE], bad[TILE];
};
// Staged partners.  Mixed forms: the endpoint's high and low parts (or, in a
// box, its fixed-point words) with the weight's mantissa parts in the fourth
// places; FP64: coordinates and the weight's 64-bit mantissa.
template <bool F64>
struct Partners;
template <>
struct Partners<false> {
  float4 h[PROB_CHUNK], l[PROB_CHUNK];
  int e[PROB_CHUNK];
};
template <>
struct Partners<true> {
  double x[PROB_CHUNK], y[PROB_CHUNK], z[PROB_CHUNK];
  unsigned long long m[PROB_CHUNK];
  int e[PROB_CHUNK];
};
template <bool F64>
struct ProbSmem {
  Partners<F64> part;
  SumSlot<F64> warp[PROB_WARPS];
  SumSlot<F64> cta[PROB_MAX_CL];  // in the cluster's first CTA
  double base[3][TILE];
};

// y_q (row items' partners, column items' own) or mu_q
__device__ __forceinline__ xd weight_y(const Workspace &w, int q) { return xd{__ldg(w.yfm + q), __ldg(w.yfe + q)}; }
__device__ __forceinline__ xd weight_mu(const Workspace &w, int q) {
  return xd{__ldg(w.ybm + (w.N - 1 - q)), __ldg(w.ybe + (w.N - 1 - q))};
}

template <bool F64, bool PBC>
__device__ __forceinline__ void stage_partner(const Workspace &w, Partners<F64> &P, int i, int q, bool beadP, xd wt) {
  const auto ep = pairg::load_end<!F64, PBC>(w, q, beadP);
  if constexpr (F64) {
    P.x[i] = ep.x;
    P.y[i] = ep.y;
    P.z[i] = ep.z;
    P.m[i] = mant64(wt.m);
  } else {
    float h, l;
    mant_hl(wt.m, h, l);
    if constexpr (PBC) {
      P.h[i] = make_float4(__uint_as_float(ep.u.x), __uint_as_float(ep.u.y), __uint_as_float(ep.u.z), h);
      P.l[i].w = l;
    } else {
      P.h[i] = make_float4(ep.h.x, ep.h.y, ep.h.z, h);
      P.l[i] = make_float4(ep.l.x, ep.l.y, ep.l.z, l);
    }
  }
  P.e[i] = wt.e;
}
// partner i's endpoint from shared memory
template <bool F64, bool PBC>
__device__ __forceinline__ pairg::EndPt<!F64, PBC> staged_end(const Partners<F64> &P, int i) {
  pairg::EndPt<!F64, PBC> e;
  if constexpr (F64) {
    e.x = P.x[i];
    e.y = P.y[i];
    e.z = P.z[i];
  } else if constexpr (PBC) {
    const float4 h = P.h[i];
    e.u = make_uint4(__float_as_uint(h.x), __float_as_uint(h.y), __float_as_uint(h.z), 0u);
  } else {
    e.h = P.h[i];
    e.l = P.l[i];
  }
  return e;
}

// One item (all threads of the cluster's CTAs; CTA `rank` of CL).
template <int MODE, bool RC, bool PBC, int GS>
__device__ __forceinline__ void exterior_item(const Workspace &w, int item, int rank, int CL,
                                              const double *__restrict__ pos, double *__restrict__ F,
                                              const unsigned long long *T63, ProbSmem<MODE == BPIMD_FP64> &sm) {
  constexpr bool F64 = MODE == BPIMD_FP64;
  using EP = pairg::EndPt<!F64, PBC>;
  using M_t = typename std::conditional<MODE == BPIMD_MIXED32, float, double>::type;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, N = w.N;
  const bool row_item = !(item & 1);
  const int tile = row_item ? w.NT - 1 - (item >> 1) : (item >> 1);
  const int me = tile * TILE + lane;
  const int mine_q = min(me, N - 1);  // lanes past N repeat the last particle and are not stored
  const EP mine = pairg::load_end<!F64, PBC>(w, mine_q, row_item);
  const xd own_w = row_item ? weight_mu(w, mine_q) : weight_y(w, mine_q);
  const int own_e = own_w.e + w.scal_i[0];  // with the exponent of 1/(N y_N)
  const int p0 = row_item ? 0 : tile * TILE, p1 = row_item ? min(N, (tile + 1) * TILE) : N;
  // partners of a chunk: a multiple of 32, so that each warp takes whole groups of four
  const int ch = min(PROB_CHUNK, ((p1 - p0 + CL - 1) / CL + 31) & ~31), per = ch / PROB_WARPS;
  // this lane's pair factors: g(partner q) at gi0 + gstr src, src = q in the
  // forward copy, N-1-q in the backward one (clamped into the stored triangle)
  const int r = row_item ? tile * TILE + lane : N - 1 - mine_q;
  const int gi0 = (int)gbase<GS>(w, r), gstr = gstride<GS>(w);
  const M_t *gm = (const M_t *)(row_item ? w.gm : w.gbm) + gi0;
  const int *ge = (row_item ? w.ge : w.gbe) + gi0;
  PSum A[3] = {{0, NO_TERM}, {0, NO_TERM}, {0, NO_TERM}};
  int bad = 0;  // components that met a non-finite difference
  float fs[3] = {0.f, 0.f, 0.f}, fc[3] = {0.f, 0.f, 0.f};
  constexpr int G = 4;
  for (int c0 = p0 + rank * ch; c0 < p1; c0 += CL * ch) {
    const int q0 = c0 + wp * per, q1 = min(q0 + per, p1);
    M_t gmv[G];
    int gev[G];
    auto load_g = [&](int q) {
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const int qk = min(q + k, p1 - 1), src = row_item ? qk : N - 1 - max(qk, mine_q);
        gmv[k] = __ldg(gm + gstr * src);
        gev[k] = __ldg(ge + gstr * src);
      }
    };
    if (!RC && q0 < q1) load_g(q0);
    if (c0 != p0 + rank * ch) __syncthreads();  // the previous chunk is read
    for (int i = threadIdx.x; i < ch; i += PROB_THREADS)
      if (c0 + i < p1)
        stage_partner<F64, PBC>(w, sm.part, i, c0 + i, !row_item, row_item ? weight_y(w, c0 + i) : weight_mu(w, c0 + i));
    __syncthreads();
    for (int q = q0; q < q1; q += G) {
      M_t m[G];
      int e[G];
#pragma unroll
      for (int k = 0; k < G; ++k) { m[k] = gmv[k]; e[k] = gev[k]; }
      if (!RC && q + G < q1) load_g(q + G);
      unsigned long long p[G][3];
      int pe[G][3], sg[G][3], E[3] = {NO_TERM, NO_TERM, NO_TERM};
#pragma unroll
      for (int k = 0; k < G; ++k) {
        const int i = min(q + k, p1 - 1) - c0;
        const bool valid = q + k < p1 && (row_item ? q + k <= me : q + k >= me);
        const EP oth = staged_end<F64, PBC>(sm.part, i);
        const EP &eb = row_item ? mine : oth, &ea = row_item ? oth : mine;
        auto d = pairg::diff3(w, eb, ea);
        if constexpr (RC && !F64) {
          // below 2^-126 a term is zero: where every lane's is, by a bound on
          // g's exponent, the power of two is left out with the rest
          const float d2 = fmaf(d.x, d.x, fmaf(d.y, d.y, d.z * d.z));
          const bool zero = !valid || pairg::g_below(d2, (float)w.cx) > (float)(sm.part.e[i] + own_e + 128);
          if (__all_sync(0xffffffffu, zero)) continue;
          m[k] = pairg::g_of_d2<MODE>(d2, w.cx, T63, e[k]);
        } else if constexpr (RC) {
          m[k] = pairg::g_of<MODE, PBC>(w, eb, ea, w.cx, T63, e[k]);
        }
        if constexpr (F64) {
          const unsigned long long t = valid ? pow2fx::mulhi(sm.part.m[i], mant64(m[k])) : 0ull;  // value t 2^(et - 63)
          const int et = valid ? sm.part.e[i] + e[k] + 1 : NO_TERM;
          const double dc[3] = {d.x, d.y, d.z};
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            bool nonfinite;
            p[k][c] = diff_term(t, dc[c], pe[k][c], sg[k][c], nonfinite);
            bad |= (valid && nonfinite) << c;
            pe[k][c] = max(pe[k][c] + et, NO_TERM);
            E[c] = max(E[c], pe[k][c]);
          }
        } else {
          const float yh = sm.part.h[i].w, yl = sm.part.l[i].w;
          const int x = sm.part.e[i] + e[k] + own_e;
          const float sc = valid && x >= -126 ? __int_as_float((min(x, 100) + 127) << 23) : 0.0f;
          float gh, gl;
          mant_hl(m[k], gh, gl);
          const float t = yh * gh, te = fmaf(yl, gh, fmaf(yh, gl, fmaf(yh, gh, -t)));
          const float th = t * sc, tl = te * sc;
          const float dc[3] = {valid ? d.x : 0.0f, valid ? d.y : 0.0f, valid ? d.z : 0.0f};
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            const float x0 = th * dc[c];
            fc[c] += fmaf(tl, dc[c], fmaf(th, dc[c], -x0));
            two_sum(fs[c], fc[c], x0);
          }
        }
      }
      if constexpr (F64) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          PSum B{0, E[c] + 3};
#pragma unroll
          for (int k = 0; k < G; ++k) {
            const long long x = (long long)(p[k][c] >> min(E[c] - pe[k][c] + 3, 63));
            B.v += (x ^ sg[k][c]) - sg[k][c];
          }
          psum_add(A[c], B);
        }
      }
    }
    if constexpr (!F64) {  // the errors of many terms, themselves rounded at 2^-24, stay below one unit of the sum
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const float err = fc[c];
        fc[c] = 0.0f;
        two_sum(fs[c], fc[c], err);
      }
    }
  }
  SumSlot<F64> &ws = sm.warp[wp];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    if constexpr (F64) { ws.v[c][lane] = A[c].v; ws.E[c][lane] = A[c].E; }
    else { ws.s[c][lane] = fs[c]; ws.c[c][lane] = fc[c]; }
  }
  if constexpr (F64) ws.bad[lane] = bad;
  __syncthreads();
  // warp c < 3: component c of the lane's sum over `n` slots, in order
  auto add_slots = [&](const SumSlot<F64> *sl, int n, int c, long long &v, int &E, int &bd, float &s, float &cc) {
    if constexpr (F64) {
      v = 0; E = NO_TERM; bd = 0;
      for (int k = 0; k < n; ++k) { E = max(E, sl[k].E[c][lane]); bd |= sl[k].bad[lane]; }
      for (int k = 0; k < n; ++k) v += shift_in(sl[k].v[c][lane], E - sl[k].E[c][lane] + 3);
      E += 3;
    } else {
      s = 0.0f; cc = 0.0f;
      for (int k = 0; k < n; ++k) { two_sum(s, cc, sl[k].s[c][lane]); cc += sl[k].c[c][lane]; }
    }
  };
  long long v = 0;
  int E = 0, bd = 0;
  float s = 0.0f, cc = 0.0f;
  if (wp < 3) {
    add_slots(sm.warp, PROB_WARPS, wp, v, E, bd, s, cc);
  } else if (rank == 0 && wp < 6 && me < N) {
    // meanwhile warps 3..5 of the first CTA: what does not need the sums
    const int c = wp - 3;
    const double own = (row_item ? w.RP : w.R1)[4 * (size_t)me + c];
    const double nb = pos[((size_t)me * w.P + (row_item ? w.P - 2 : 1)) * 3 + c];  // bead P-1, or bead 2
    double b = img<PBC>(w, own - nb);
    if (row_item ? me + 1 < N : me >= 1) {  // the direct link me -> me+1, or me-1 -> me
      const double oth = row_item ? w.R1[4 * (size_t)(me + 1) + c] : w.RP[4 * (size_t)(me - 1) + c];
      b = fma(direct_link_fast(w, row_item ? me : me - 1), img<PBC>(w, own - oth), b);
    }
    sm.base[c][lane] = b;
  }
  if (CL > 1) {
    cluster_wait_acquire();  // every CTA of the cluster has started (it arrived at its start)
    if (wp < 3) {
      SumSlot<F64> &cs = sm.cta[rank];
      if constexpr (F64) {
        cluster_store(&cs.v[wp][lane], v);
        cluster_store(&cs.E[wp][lane], E);
        if (wp == 0) cluster_store(&cs.bad[lane], bd);
      } else {
        cluster_store(&cs.s[wp][lane], s);
        cluster_store(&cs.c[wp][lane], cc);
      }
    }
    cluster_arrive_release();
    cluster_wait_acquire();
    if (rank == 0 && wp < 3) add_slots(sm.cta, CL, wp, v, E, bd, s, cc);
  } else {
    __syncthreads();
  }
  if (rank == 0 && wp < 3 && me < N) {
    const double mz = own_w.m * w.scal[1];
    double W;
    if constexpr (F64) {
      W = ((double)v * mz) * pow2_normal(E - 61 + own_e);
      if ((bd >> wp) & 1) W = __longlong_as_double(0x7ff8000000000000LL);
    } else {
      W = ((double)s + (double)cc) * mz;
    }
    const double f = -w.k * (sm.base[wp][lane] + (row_item ? W : -W));
    F[((size_t)me * w.P + (row_item ? w.P - 1 : 0)) * 3 + wp] = f;
    if (!isfinite(f)) atomicOr(w.status, ST_NONFINITE);
  }
}

// CL CTAs (one cluster) per item
template <int MODE, bool RC>
__global__ void __launch_bounds__(PROB_THREADS) exterior_kernel(Workspace w, const double *__restrict__ pos,
                                                                double *__restrict__ F, int CL) {
  __shared__ ProbSmem<MODE == BPIMD_FP64> sm;
  __shared__ unsigned long long T63[RC ? 256 : 1];
  if (CL > 1) cluster_arrive_release();
  if (RC && MODE != BPIMD_MIXED32) {
    pairg::table_init(T63);
    __syncthreads();
  }
  pdl_wait();
  const int item = blockIdx.x / CL, rank = blockIdx.x % CL;
  if (w.pbc) exterior_item<MODE, RC, true, 0>(w, item, rank, CL, pos, F, T63, sm);
  else exterior_item<MODE, RC, false, 0>(w, item, rank, CL, pos, F, T63, sm);
  pdl_trigger();
}

// Replica batch: entry k of tab is (replica, item); positions and forces of
// replica r start at element off[r] of the packed arrays.
template <int MODE>
__global__ void __launch_bounds__(PROB_THREADS) exterior_batched(const Workspace *__restrict__ ws,
                                                                 const int2 *__restrict__ tab, int ntab,
                                                                 const long long *__restrict__ off,
                                                                 const double *__restrict__ pos,
                                                                 double *__restrict__ F) {
  __shared__ ProbSmem<MODE == BPIMD_FP64> sm;
  pdl_wait();
  for (int k = blockIdx.x; k < ntab; k += gridDim.x) {
    const int2 e = tab[k];
    exterior_item<MODE, false, false, 32>(ws[e.x], e.y, 0, 1, pos + off[e.x], F + off[e.x], nullptr, sm);
    __syncthreads();  // the slots are read
  }
  pdl_trigger();
}

// Sum over the block's threads (fixed order); thread 0 gets it.
__device__ double sum_block(double v, double *red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double sum = 0.0;
  if (threadIdx.x == 0)
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) sum += red[q];
  __syncthreads();
  return sum;
}

// Expected spring energy over representative permutations, in parts: block blk
// of the lower triangle gives (1/2) m w_P^2 sum_{a<=b in block} Pr[b -> a]
// |r_b^P - r_a^1|^2, and particles 256 blk .. 256 blk + 255 their interior
// springs and direct links.  Float64 throughout; run once per
// molecular-dynamics call, for the primitive energy estimator.  The exponents
// of a probability's factors are added first: below 2^-100 it adds nothing to a
// sum of order N kT, and its float64 arithmetic (~75 cycles an instruction, ~30
// of them) and loads are left out -- nearly every pair of a liquid (391 us a
// call at N = 4000 before).  All threads of the block call it; thread 0 gets the sum.
__device__ double spring_block(const Workspace &w, int blk, double *red) {
  int t, s;
  block_coords_f(blk, t, s);
  const int inv_e = w.scal_i[0];
  const double inv_m = w.scal[1];
  double acc = 0.0;
  for (int e = threadIdx.x; e < TILE2; e += blockDim.x) {
    const int a = s * TILE + (e >> 5), b = t * TILE + (e & 31);
    if (b < w.N && a <= b) {
      const size_t gi = gbase(w, b) + w.gstr * a;
      const int r = w.N - 1 - b;
      int ex = w.yfe[a] + w.ybe[r] + inv_e;
      xd g{0.0, 0};
      if (w.recomp) g = pairg::g_runtime(w, a, b);
      else g.e = w.ge[gi];
      ex += g.e;
      if (ex >= -100) {
        if (!w.recomp) g.m = w.mixed ? (double)((const float *)w.gm)[gi] : ((const double *)w.gm)[gi];
        const double M = (w.yfm[a] * w.ybm[r]) * (g.m * inv_m) * pow2_normal(ex);
        const double dx = mimage(w, w.RP[4 * b] - w.R1[4 * a]), dy = mimage(w, w.RP[4 * b + 1] - w.R1[4 * a + 1]),
                     dz = mimage(w, w.RP[4 * b + 2] - w.R1[4 * a + 2]);
        acc += M * (dx * dx + dy * dy + dz * dz);
      }
    }
  }
  acc *= w.half_k;
  const int l = blk * blockDim.x + threadIdx.x;
  if (l < w.N) {
    acc += w.Eint[l];
    if (l + 1 < w.N) acc += direct_link_fast(w, l) * w.link[l];
  }
  return sum_block(acc, red);
}

__global__ void __launch_bounds__(256) spring_expect_kernel(Workspace w, double *part) {
  __shared__ double red[8];
  for (int blk = blockIdx.x; blk < w.NB; blk += gridDim.x) {
    const double v = spring_block(w, blk, red);
    if (threadIdx.x == 0) part[blk] = v;
  }
}

// Replica batch: entry k of tab is (replica, block); part[k] as above, and
// part[ntab + k] the sum of v^2 over the block's share of the replica's
// velocities (packed, replica r at element off[r]).
__global__ void __launch_bounds__(256) spring_expect_batched(const Workspace *__restrict__ ws,
                                                             const int2 *__restrict__ tab, int ntab,
                                                             const long long *__restrict__ off,
                                                             const double *__restrict__ vel, double *part) {
  __shared__ double red[8];
  for (int k = blockIdx.x; k < ntab; k += gridDim.x) {
    const int2 e = tab[k];
    const Workspace &w = ws[e.x];
    const double v = spring_block(w, e.y, red);
    const long long n = 3LL * w.N * w.P, lo = n * e.y / w.NB, hi = n * (e.y + 1) / w.NB;
    double ke = 0.0;
    for (long long i = lo + threadIdx.x; i < hi; i += blockDim.x) ke = fma(vel[off[e.x] + i], vel[off[e.x] + i], ke);
    ke = sum_block(ke, red);
    if (threadIdx.x == 0) {
      part[k] = v;
      part[ntab + k] = ke;
    }
  }
}

__global__ void dense_prob_kernel(Workspace w, double *M) {
  const size_t NN = (size_t)w.N * w.N;
  for (size_t idx = blockIdx.x * (size_t)blockDim.x + threadIdx.x; idx < NN; idx += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(idx / w.N), a = (int)(idx % w.N);  // row l = b, column l' = a
    double v = 0.0;
    if (a <= b) {
      const size_t gi = gbase(w, b) + w.gstr * a;
      const xd g = w.recomp ? pairg::g_runtime(w, a, b)
                            : xd{w.mixed ? (double)((const float *)w.gm)[gi] : ((const double *)w.gm)[gi], w.ge[gi]};
      const xd al = alpha_of(w, a), mu = mu_of(w, b);
      v = xtod(xd{al.m * mu.m * g.m, al.e + mu.e + g.e});
    } else if (a == b + 1) {
      v = direct_link_prob(w, b);
    }
    M[idx] = v;
  }
}

}  // namespace

namespace {
template <int MODE, bool RC>
cudaError_t launch_exterior(const Workspace &w, const double *pos, double *F, cudaStream_t s) {
  // CTAs per item: enough that a warp has a few groups of four partners (the
  // longest list is N), few enough that the cluster barrier and the staging do
  // not outweigh them.  Whole evaluation, mixed, with 1 / 2 / 4 / 8 CTAs: N = 64
  // 23.0 / 22.7 / 22.4 / 22.4 us, N = 256 34.0 / 32.2 / 31.2 / 31.0, N = 1024
  // 84.8 / 75.1 / 71.9 / 72.8, N = 1601 138 / 126 / 123 / 120, N = 4096
  // 502 / 477 / 470 / 478 (past ~64 tiles four fill the GPU).
  const int CL = w.NT <= 1 ? 1 : w.NT <= 2 ? 2 : w.NT <= 32 ? 4 : w.NT <= 64 ? 8 : 4;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * w.NT * CL);
  cfg.blockDim = dim3(PROB_THREADS);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CL;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, exterior_kernel<MODE, RC>, w, pos, F, CL);
}
}  // namespace

cudaError_t launch_prob_forces(const Workspace &w, const double *pos, double *F, cudaStream_t s) {
  switch (w.mode) {
    case BPIMD_FP64:
      return w.recomp ? launch_exterior<BPIMD_FP64, true>(w, pos, F, s) : launch_exterior<BPIMD_FP64, false>(w, pos, F, s);
    case BPIMD_MIXED:
      return w.recomp ? launch_exterior<BPIMD_MIXED, true>(w, pos, F, s) : launch_exterior<BPIMD_MIXED, false>(w, pos, F, s);
    default:
      return w.recomp ? launch_exterior<BPIMD_MIXED32, true>(w, pos, F, s)
                      : launch_exterior<BPIMD_MIXED32, false>(w, pos, F, s);
  }
}

cudaError_t launch_spring_expectation(const Workspace &w, double *part, cudaStream_t s) {
  const int sms = sm_count();
  const int grid = w.NB < sms * 8 ? w.NB : sms * 8;
  spring_expect_kernel<<<grid, 256, 0, s>>>(w, part);
  return cudaGetLastError();
}

cudaError_t launch_spring_expectation_batched(const Workspace *ws, const int2 *tab, int ntab, const long long *off,
                                             const double *vel, double *part, cudaStream_t s) {
  if (ntab <= 0) return cudaSuccess;
  const int sms = sm_count();
  const int grid = ntab < sms * 8 ? ntab : sms * 8;
  spring_expect_batched<<<grid, 256, 0, s>>>(ws, tab, ntab, off, vel, part);
  return cudaGetLastError();
}

cudaError_t launch_dense_probabilities(const Workspace &w, double *M, cudaStream_t s) {
  dense_prob_kernel<<<1024, 256, 0, s>>>(w, M);
  return cudaGetLastError();
}

cudaError_t launch_prob_forces_batched(const Workspace *ws, const int2 *tab, int ntab, const long long *off,
                                      int mode, const double *pos, double *F, int blocks_per_sm, cudaStream_t s) {
  if (ntab <= 0) return cudaSuccess;
  const int sms = sm_count();
  const int cap = sms * (blocks_per_sm > 0 ? blocks_per_sm : 8);
  const int grid = ntab < cap ? ntab : cap;
  cudaError_t e;
  switch (mode) {
    case BPIMD_FP64: e = launch_pdl(exterior_batched<BPIMD_FP64>, grid, 256, 0, s, ws, tab, ntab, off, pos, F); break;
    case BPIMD_MIXED: e = launch_pdl(exterior_batched<BPIMD_MIXED>, grid, 256, 0, s, ws, tab, ntab, off, pos, F); break;
    default: e = launch_pdl(exterior_batched<BPIMD_MIXED32>, grid, 256, 0, s, ws, tab, ntab, off, pos, F); break;
  }
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace bpimd
