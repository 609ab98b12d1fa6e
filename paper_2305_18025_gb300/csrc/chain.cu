// Forward and backward potential recursions as blocked triangular solves.
//
// Forward  (Eq. our-forward-potential-recurrence, linear-space form):
//   y_0 = 1,  y_{r+1} = c_{r+1} * S_r,  S_r = sum_{w<=r} y_w g(w+1, r+1)
// Backward (Eq. backward-potential-recursion, linear-space form), with rows
// r = N-1-a and sources w = N-1-b so that it has the same lower-triangular
// shape:  Y_0 = mu_N = 1, S_r = B_{a+1} = sum_{w<=r} Y_w g(a+1, b+1),
//   Y_{r+1} = mu_a = c_a * S_r   (c_0 := 1 for the last row, Y_N = B_1).
// Both read  Y_{r+1} = c_r sum_{w<=r} H(w, r) Y_w  with the pair factors H of
// the recursion's own coordinates and c_r its row coefficient.
//
// Panels.  Panel t (rows r = 64t + j) has the unknowns X^t_j = Y_{64t+1+j}.
//   X^t = b^t + L^t X^t,      L^t(j, i) = c_r H(64t+1+i, r)  for i < j,
//   b^t_j = c_r (A^t_j + sum_i H(64t-63+i, r) X^{t-1}_i),
// where A^t_j sums the sources before X^{t-1}.  Hence
//   X^t = M^t b^t,   M^t = (I - L^t)^{-1} = sum_k (L^t)^k,
// a unit lower-triangular matrix with nonnegative entries, so every sum below
// adds nonnegative terms: no cancellation anywhere.  M^t depends on the
// positions only: panel_inverse_kernel forms it for every panel at once.  The
// sequential part is two matrix-vector products a panel.
//
// Cluster schedule (chain_kernel).  One cluster a recursion; CTA q owns rows
// q R .. q R + R-1 of every panel (R = 64 / cluster size).  Its critical warps
// (one row each, two products a lane) form their rows of b^t from
// X^{t-1}, store them into every CTA's shared memory (st.async, counted on an
// mbarrier there), wait for all of b^t, form their rows of X^t = M^t b^t and
// hand those round the same way: two exchanges of 64 values a panel and no
// cluster barrier.  Operands (rows of c H and M) are loaded a panel ahead.
// The other warps add X^t to the sums A of their rows in panels t+2 and later
// (one warp a panel; the panel the critical warps need next comes first), each
// lane keeping its own partial sum, which the critical warps reduce with the
// panel's own products.  Every value is an extended number m 2^e on 64-bit
// integer mantissas (the xi format of chain_common.cuh): GB300's float64 pipe
// retires ~1.7 lanes a clock, with a 64-cycle latency.  Every wait is bounded.
// Slots: X has one a panel; b has two, and b^{t+2} is sent only after X^{t+1}
// is complete, i.e. after every CTA has read b^{t+1}, and b^t before it.
//
// Superblocks.  A chain launch takes up to MAX_PANELS panels.  Between two
// launches source_update_kernel, spread over the whole GPU, adds the finished
// superblock's Y to the sums of every later row.
#include <cooperative_groups.h>
#include <mutex>
#include <type_traits>

#include "chain_common.cuh"

namespace cg = cooperative_groups;

namespace bpimd {
namespace {

using namespace chain_detail;

constexpr int PT = CHAIN_PANEL;  // rows of a panel
static_assert(PT == 2 * TILE, "a panel inverse joins two tile inverses");
constexpr int MAX_PANELS = 32;   // panels of one chain launch
constexpr int SLICES = CHAIN_SLICES;  // partial sums a row carries from superblock to superblock
constexpr int PINV_THREADS = 512;

// Panels of one chain launch.  One launch while its clusters keep up with the
// sums of later panels; past that, equal superblocks of at most 16 panels, the
// whole GPU adding each to the later rows.  Evaluations, one launch /
// superblocks: N = 1601 103.4 / 106.3 us, N = 2048 133.8 / 130.2.  With 16 / 12 /
// 8 panels a superblock: N = 4096 349 / 364 / 377, recomputed factors N = 8788
// 1024 / 1042 / 1092, N = 16384 2787 / 2878 / 2989.
inline int superblock_panels(int panels, bool RC) {
  if (panels <= (RC ? 16 : 28)) return panels;
  const int k = (panels + 15) / 16;
  return (panels + k - 1) / k;
}

// Panel t's inverse M of one recursion, [row][column].
__device__ __forceinline__ size_t panel_base(const Workspace &w, bool bwd, int t) {
  return (size_t)((bwd ? (w.N + PT - 1) / PT : 0) + t) * PT * PT;
}

// acc += sum_i H(src + i STRIDE, row) y_i over eight sources, H recomputed.
// The exponents come first: where every lane's eight terms lie below 2^-64 of
// its sum they would be shifted out of it, and the powers of two (the larger
// part of the work) are left out.  The sum's bits are the same.
template <int MODE, bool BWD, bool PBC, int STRIDE>
__device__ __forceinline__ void add_sources_rc(const Workspace &w, const RowFactors<MODE, BWD, true, PBC> &f, bool row_ok,
                                               int src, int last, const xi (&y)[8], const unsigned long long *T63,
                                               xi &acc) {
  using M_t = typename std::conditional<MODE == BPIMD_MIXED32, float, double>::type;
  using D_t = typename std::conditional<MODE == BPIMD_FP64, double, float>::type;
  D_t d2[8];
  bool need = false;
  const float cxf = (float)w.cx;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    d2[i] = f.re.dist2(w, min(src + STRIDE * i, last));
    // pe = e + y.e + 1 with e <= -floor(gap); the eight terms add three bits
    need |= !(pairg::g_below(d2[i], cxf) > (float)(y[i].e - acc.e + 70));
  }
  if (!__any_sync(0xffffffffu, need && row_ok)) return;
  unsigned long long kk[8];
  int e[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const M_t m = pairg::g_of_d2<MODE>(d2[i], w.cx, T63, e[i]);
    kk[i] = mant53(m) << 11;
  }
  if (row_ok) acc = xi_add(acc, xsum_fin<3>(xsum_dot<3, 8>(kk, e, y, 0, 2 * XZERO_E)));
}

// ---------------------------------------------------------- panel inverses
// A panel and recursion: a cluster of four CTAs.  The CTA pair of diagonal
// tile q / 2 inverts it, each CTA every other column: thread (i, j) forms
// L(j, i); then a warp forms column k by forward substitution, lane j holding
// M(j, k), step s adding L(j, s) M(s, k) once M(s, k) is final, and stores it
// into all four CTAs.  With the tiles' inverses M1 and M2 there, the block
// below the diagonal is M21 = M2 (L21 M1): each CTA forms eight of its
// columns, two lanes an entry, leaving out the zeros of the triangles.  The
// kernel is bound by the integer pipe's multiplications (~50 issue cycles a
// product and aligned addition), hence four SMs a panel: one CTA a tile and
// two a panel took 16 us a launch at N = 1024.
struct PinvSmem {
  unsigned long long Lk[TILE][TILE], L21k[TILE][TILE];  // [source][row]
  unsigned long long M1m[TILE][TILE], M2m[TILE][TILE];  // [column][row], xi format
  unsigned long long Tm[8][TILE];                       // [column][row]
  int Le[TILE][TILE], L21e[TILE][TILE], M1e[TILE][TILE], M2e[TILE][TILE], Te[8][TILE];
  unsigned long long T63[256];
};

template <int MODE, bool BWD, bool RC, bool PBC>
__device__ void panel_inverse_body(const Workspace &w, int t, int q, PinvSmem &sm) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, tile = q >> 1;
  const int r0 = t * PT, row = r0 + tile * TILE + lane, row1 = r0 + TILE + lane;
  const bool two = r0 + TILE < w.N;  // the second tile has rows
  // the tile's own L (source i of it), and L21 (source i of tile 0, rows of tile 1)
  {
    RowFactors<MODE, BWD, RC, PBC> f, f1;
    xd c{1.0, XZERO_E}, c1 = c;
    if (row < w.N) { f.load(w, row); c = xnorm_int(chain_coef<BWD>(w, row)); }
    if (row1 < w.N) { f1.load(w, row1); c1 = xnorm_int(chain_coef<BWD>(w, row1)); }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int i = wid + 16 * h;
      xk L{1ull << 63, XZERO_E}, L21{1ull << 63, XZERO_E};
      if (row < w.N && i < lane) L = f.k(w, c, r0 + tile * TILE + 1 + i, sm.T63);
      if (row1 < w.N) L21 = f1.k(w, c1, r0 + 1 + i, sm.T63);
      sm.Lk[i][lane] = L.m;
      sm.Le[i][lane] = L.e;
      sm.L21k[i][lane] = L21.m;
      sm.L21e[i][lane] = L21.e;
    }
  }
  __syncthreads();
  const int k = 2 * wid + (q & 1);
  xi acc{1ull << 62, lane == k ? 0 : XZERO_E};
  if (tile == 0 || two)
    for (int s = k; s < TILE - 1; ++s) {
      xi y;
      y.m = __shfl_sync(0xffffffffu, acc.m, s);
      y.e = __shfl_sync(0xffffffffu, acc.e, s);
      acc = xi_fma(acc, sm.Lk[s][lane], sm.Le[s][lane], y);
    }
  cg::cluster_group cluster = cg::this_cluster();
  const size_t base = panel_base(w, BWD, t);
  unsigned long long *gk = w.bk + base;
  int *gke = w.be + base;
  unsigned long long *Mm = tile == 0 ? &sm.M1m[k][lane] : &sm.M2m[k][lane];
  int *Me = tile == 0 ? &sm.M1e[k][lane] : &sm.M2e[k][lane];
  cluster_wait();
#pragma unroll
  for (int o = 0; o < 4; ++o) {
    *cluster.map_shared_rank(Mm, o) = acc.m;
    *cluster.map_shared_rank(Me, o) = acc.e;
  }
  cluster.sync();
  // rows 16 q .. 16 q + 15 of the panel's inverse, but for the block M21 (K
  // format: twice the xi mantissa is the same value)
  {
    const int j = 16 * (q & 1) + wid, r = tile * TILE + j;
    gk[r * PT + tile * TILE + lane] = (tile == 0 ? sm.M1m[lane][j] : sm.M2m[lane][j]) << 1;
    gke[r * PT + tile * TILE + lane] = tile == 0 ? sm.M1e[lane][j] : sm.M2e[lane][j];
    if (tile == 0 || !two) {
      gk[r * PT + (1 - tile) * TILE + lane] = 1ull << 63;
      gke[r * PT + (1 - tile) * TILE + lane] = XZERO_E;
    }
  }
  if (!two) return;
  // T = L21 M1, then M21 = M2 T, column col = 4 (wid / 2) + q; warp: rows
  // 16 (wid % 2) .. +15, lane: row j, the sum's terms h, h + 2, ... of each group of eight
  const int slot = wid >> 1, col = 4 * slot + q, j = 16 * (wid & 1) + (lane >> 1), h = lane & 1;
  auto dot = [&](int g0, int g1, auto kk, auto ke, auto ym, auto ye) {
    xsum sum{0, 2 * XZERO_E};
    for (int g = g0; g < g1; ++g) {
      unsigned long long a[4];
      int ae[4];
      xi y[4];
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        const int x = 8 * g + 2 * n + h;
        a[n] = kk(x);
        ae[n] = ke(x);
        y[n] = xi{ym(x), ye(x)};
      }
      sum = xsum_add(sum, xsum_dot<5, 4>(a, ae, y, 0, 2 * XZERO_E));
    }
    xsum u;
    u.s = __shfl_xor_sync(0xffffffffu, sum.s, 1);
    u.E = __shfl_xor_sync(0xffffffffu, sum.E, 1);
    sum = xsum_add(sum, u);
    return sum.s ? xsum_fin<5>(sum) : xi{1ull << 62, XZERO_E};
  };
  const xi T = dot(col >> 3, 4, [&](int x) { return sm.L21k[x][j]; }, [&](int x) { return sm.L21e[x][j]; },
                   [&](int x) { return sm.M1m[col][x]; }, [&](int x) { return sm.M1e[col][x]; });
  if (h == 0) {
    sm.Tm[slot][j] = T.m;
    sm.Te[slot][j] = T.e;
  }
  __syncthreads();
  const xi m21 = dot(0, 2 + 2 * (wid & 1), [&](int x) { return sm.M2m[x][j] << 1; }, [&](int x) { return sm.M2e[x][j]; },
                     [&](int x) { return sm.Tm[slot][x]; }, [&](int x) { return sm.Te[slot][x]; });
  if (h == 0) {
    gk[(TILE + j) * PT + col] = m21.m << 1;
    gke[(TILE + j) * PT + col] = m21.e;
  }
}

template <int MODE, bool RC>
__global__ void __launch_bounds__(PINV_THREADS) __cluster_dims__(4, 1, 1) panel_inverse_kernel(Workspace w) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PinvSmem &sm = *(PinvSmem *)smem_raw;
  cluster_arrive();  // waited for before the first store into another CTA
  if (RC) {
    pairg::table_init(sm.T63);
    __syncthreads();
  }
  pdl_wait();
  pdl_trigger();  // the recursions wait for this grid's completion
  const int t = blockIdx.x >> 2, q = blockIdx.x & 3;
  const bool bwd = blockIdx.y != 0;
  if (w.pbc) {
    if (bwd) panel_inverse_body<MODE, true, RC, true>(w, t, q, sm);
    else panel_inverse_body<MODE, false, RC, true>(w, t, q, sm);
  } else {
    if (bwd) panel_inverse_body<MODE, true, RC, false>(w, t, q, sm);
    else panel_inverse_body<MODE, false, RC, false>(w, t, q, sm);
  }
}

// ------------------------------------------------------------ recursions
// A value handed round a cluster: one 16-byte store.
struct __align__(16) Wire {
  unsigned long long m;
  int e, pad;
};

struct ChainSmem {
  Wire X[MAX_PANELS][PT];               // the superblock's unknowns, by panel
  Wire b[2][PT];                        // b of panel t in slot t & 1
  unsigned long long Am[MAX_PANELS][32];  // partial sums A of this CTA's rows: lane (source part) * R + row
  int Ae[MAX_PANELS][32];
  unsigned long long xbar[MAX_PANELS];  // X^t has arrived
  unsigned long long bbar[MAX_PANELS];  // b^t has arrived
  unsigned long long done[MAX_PANELS];  // A of panel t is complete up to X^{t-2}
  unsigned long long never;             // an mbarrier nothing arrives on (BPIMD_FLAG_TEST_TIMEOUT)
  unsigned long long T63[256];          // recompute mode
  double misc[2];                       // end of the forward recursion: C'[N]
  long long nsum;
  int aborted;                          // a hand-off wait of this CTA expired
};

__device__ __forceinline__ void st_async_wire(unsigned raddr, xi v, unsigned rbar) {
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(raddr),
               "r"((unsigned)v.m), "r"((unsigned)(v.m >> 32)), "r"((unsigned)v.e), "r"(0u), "r"(rbar)
               : "memory");
}
__device__ __forceinline__ xi wire_get(const Wire *p) {
  const ulonglong2 v = *(const ulonglong2 *)p;
  return xi{v.x, (int)v.y};
}

// A row's sum over a warp: two products a lane (kk y, in the K and xi formats)
// and one more term (p0, pe0) a lane, at most 72 terms in all.  The largest
// exponent first (one redux), then every term aligned to it with two bits of
// headroom for the lane's three (2^-59 of the largest), and the 63-bit sums added
// exactly in three pieces of 21 bits by redux: four warp-wide steps where a
// shuffle tree of extended numbers takes five levels of six.
__device__ __forceinline__ xi row_sum(const unsigned long long (&kk)[2], const int (&ke)[2], const xi (&y)[2],
                                      unsigned long long p0, int pe0) {
  unsigned long long p[2];
  int pe[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    p[i] = pow2fx::mulhi(kk[i], y[i].m);
    pe[i] = ke[i] + y[i].e + 1;
  }
  const int E = __reduce_max_sync(0xffffffffu, max(pe0, max(pe[0], pe[1])));
  const unsigned long long s =
      (p0 >> min(E - pe0 + 2, 63)) + (p[0] >> min(E - pe[0] + 2, 63)) + (p[1] >> min(E - pe[1] + 2, 63));
  const unsigned lo = __reduce_add_sync(0xffffffffu, (unsigned)s & 0x1FFFFFu);
  const unsigned mid = __reduce_add_sync(0xffffffffu, (unsigned)(s >> 21) & 0x1FFFFFu);
  const unsigned hi = __reduce_add_sync(0xffffffffu, (unsigned)(s >> 42));
  // hi 2^42 + mid 2^21 + lo < 2^68: five bits less of it where it would not fit
  const int k = hi >> 20 ? 5 : 0;
  return xsum_fin<2>(xsum{((unsigned long long)hi << (42 - k)) + ((((unsigned long long)mid << 21) + lo) >> k), E + k});
}

template <int CL>
struct ChainShape {
  static constexpr int R = PT / CL;            // rows of a panel a CTA owns
  static constexpr int CRIT = R;               // critical warps (one row each)
  static constexpr int PARTS = 32 / R;         // source parts of a bulk task (lanes a row)
  static constexpr int SRC = PT / PARTS;       // sources a lane of a bulk task
  static constexpr int BULK = 14;              // bulk warps
  static constexpr int THREADS = 32 * (CRIT + BULK + 1);  // one more warp: the prefix sums
};

// MODE: precision form (the stored-factor kernels serve BPIMD_MIXED with the
// BPIMD_FP64 code: the same float64-mantissa layout); RC: recompute mode, H
// formed from the endpoint copies wherever it is used.  Panels t0 .. t0+np-1.
template <int MODE, bool BWD, int CL, bool RC, bool PBC>
__device__ void run_chain(const Workspace &w, int t0, int np, ChainSmem &sm, double *V_B) {
  using S = ChainShape<CL>;
  constexpr int R = S::R, PARTS = S::PARTS, SRC = S::SRC;
  using M_t = typename std::conditional<MODE == BPIMD_MIXED32, float, double>::type;
  const unsigned rank = cg::this_cluster().block_rank();
  const int N = w.N, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int row0 = t0 * PT;  // first row of the superblock
  double *gYm = BWD ? w.ybm : w.yfm;
  int *gYe = BWD ? w.ybe : w.yfe;
  volatile int *aborted = (volatile int *)&sm.aborted;

  if (tid < np) {
    mbar_init(smem_addr(&sm.xbar[tid]), 1);
    mbar_init(smem_addr(&sm.bbar[tid]), 1);
    mbar_init(smem_addr(&sm.done[tid]), 1);
    mbar_fence_init();
    // one use a launch: the 64 values of a panel are expected from the start
    mbar_expect_tx(smem_addr(&sm.xbar[tid]), PT * sizeof(Wire));
    mbar_expect_tx(smem_addr(&sm.bbar[tid]), PT * sizeof(Wire));
  }
  if (tid == 0) {
    mbar_init(smem_addr(&sm.never), 1);
    mbar_fence_init();
    sm.aborted = 0;
  }
  if (RC) pairg::table_init(sm.T63);
  // the set-up above touches shared memory only: it runs, and the cluster
  // barrier starts, before the preceding grid is complete
  __syncthreads();
  cluster_arrive();
  pdl_wait();
  // After the wait, never before it: what is launched to run beside this kernel
  // (the physical force, later rows' updates) starts here without a wait of its
  // own, and what needs the recursions waits for this grid.
  pdl_trigger();
  if (t0 == 0 && rank == 0 && tid == 0) {
    gYm[0] = 1.0;
    gYe[0] = 0;
    if (!BWD) w.C[0] = 0.0;
  }
  // the sums the panels start from: H(0, r) Y_0, or the earlier superblocks' sums
  for (int x = tid; x < np * 32; x += S::THREADS) {
    const int p = x >> 5, part = (x & 31) / R, r = row0 + p * PT + (int)rank * R + (x & 31) % R;
    xi a{1ull << 62, XZERO_E};
    if (r < N) {
      if (t0 == 0) {
        if (part == 0) {
          RowFactors<MODE, BWD, RC, PBC> f;
          f.load(w, r);
          M_t m;
          int e;
          f.h(w, 0, sm.T63, m, e);
          a = xi{mant53(m) << 10, e};
        }
      } else if (part < SLICES) {
        const size_t k = ((size_t)(BWD ? SLICES : 0) + part) * N + r;
        a = xi{w.Asm[k], w.Ase[k]};
      }
    }
    sm.Am[p][x & 31] = a.m;
    sm.Ae[p][x & 31] = a.e;
  }
  __syncthreads();
  cluster_wait();  // every mbarrier of the cluster is initialised

  if (wid < S::CRIT) {
    if (!BWD && w.test_timeout && rank == 0) handoff_wait(smem_addr(&sm.never), 0, w.status, aborted);
    const int prow = (int)rank * R + wid;  // row of the panel
    // where this lane's copies of a row's value go (panel p: + p or p & 1 slots)
    const int dest = lane < CL ? lane : 0;
    const unsigned bdst = cluster_addr(smem_addr(&sm.b[0][prow]), dest), xdst = cluster_addr(smem_addr(&sm.X[0][prow]), dest);
    const unsigned bbardst = cluster_addr(smem_addr(&sm.bbar[0]), dest), xbardst = cluster_addr(smem_addr(&sm.xbar[0]), dest);
    const unsigned bbar = smem_addr(&sm.bbar[0]), xbar = smem_addr(&sm.xbar[0]), done = smem_addr(&sm.done[0]);
    // Operands: loaded a panel ahead, made ready (c H, c A) while the values
    // of the panel before are on their way round the cluster, so that nothing
    // but products and exchanges is on the path from X^{p-1} to X^p.
    xd craw{1.0, XZERO_E}, c{1.0, XZERO_E};
    unsigned long long Mk[2], Mnext[2] = {0, 0}, Hk[2] = {0, 0};
    int Me[2], Menext[2] = {0, 0}, He[2] = {XZERO_E, XZERO_E};
    M_t hm[2];
    int he[2];
    xi ca{0, 2 * XZERO_E};
    bool ok = true;
    auto load_m = [&](int p) {
      const size_t base = panel_base(w, BWD, t0 + p) + (size_t)prow * PT + lane;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        Mnext[k] = __ldg(w.bk + base + 32 * k);
        Menext[k] = __ldg(w.be + base + 32 * k);
      }
    };
    auto load_row = [&](int p) {  // c and H of the previous panel's unknowns, columns lane and lane + 32
      const int r = row0 + p * PT + prow;
      craw = xd{1.0, XZERO_E};
      if (r < N) craw = chain_coef<BWD>(w, r);
      if (p == 0) return;
      RowFactors<MODE, BWD, RC, PBC> f;
      f.load(w, min(r, N - 1));
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        hm[k] = (M_t)1.0;
        he[k] = XZERO_E;
        if (r < N) f.h(w, row0 + p * PT - PT + 1 + lane + 32 * k, sm.T63, hm[k], he[k]);
      }
    };
    auto ready_row = [&](int p) {
      c = xnorm_int(craw);
      if (p == 0) return;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const xk x = mul_mant<M_t>(c, hm[k], he[k]);
        Hk[k] = x.m;
        He[k] = x.e;
      }
    };
    auto ready_sum = [&](int p) {  // c A: this lane's partial sum of the row, complete up to X^{p-2}
      if (p >= 2) ok &= handoff_wait(done + 8 * p, 0, w.status, aborted);
      if (lane < PARTS) ca = xi_mul(xi{sm.Am[p][lane * R + wid], sm.Ae[p][lane * R + wid]}, c);
    };
    load_row(0);
    load_m(0);
    ready_row(0);
    ready_sum(0);
    if (np > 1) load_row(1);
    xi X[2] = {{0, XZERO_E}, {0, XZERO_E}};
    for (int p = 0; p < np; ++p) {
#pragma unroll
      for (int k = 0; k < 2; ++k) { Mk[k] = Mnext[k]; Me[k] = Menext[k]; }
      if (p + 1 < np) load_m(p + 1);
      // b_j = c_j (A_j + sum_i H(j, i) X^{p-1}_i): 64 products and up to 8 partial sums
      const xi b = row_sum(Hk, He, X, ca.m, ca.e);
      if (lane < CL && ok) st_async_wire(bdst + (p & 1) * (unsigned)sizeof(sm.b[0]), b, bbardst + 8 * p);
      if (p + 1 < np) {
        ready_row(p + 1);
        if (p + 2 < np) load_row(p + 2);
      }
      // X_j = sum_{i <= j} M(j, i) b_i
      ok &= handoff_wait(bbar + 8 * p, 0, w.status, aborted);
      xi B[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) B[k] = wire_get(&sm.b[p & 1][lane + 32 * k]);
      const xi x = row_sum(Mk, Me, B, 0, 2 * XZERO_E);
      if (lane < CL && ok) st_async_wire(xdst + p * (unsigned)sizeof(sm.X[0]), x, xbardst + 8 * p);
      if (p + 1 < np) ready_sum(p + 1);
      const int r = row0 + p * PT + prow;
      if (lane == 0 && r < N) {
        const xd y = xi_to_xd(x);
        gYm[r + 1] = y.m;
        gYe[r + 1] = y.e;
      }
      ok &= handoff_wait(xbar + 8 * p, 0, w.status, aborted);
      if (p + 1 < np)
#pragma unroll
        for (int k = 0; k < 2; ++k) X[k] = wire_get(&sm.X[p][lane + 32 * k]);
    }
  } else if (wid < S::CRIT + S::BULK) {
    // bulk warp bw: panels p = bw, bw + BULK, ...; in period t (X^t) those from t + 2
    const int bw = wid - S::CRIT, rr = lane % R, part = lane / R;
    auto first_panel = [&](int t) { return t + 2 + ((bw - (t + 2)) % S::BULK + S::BULK) % S::BULK; };
    M_t fm[SRC];
    int fe[SRC];
    auto load_factors = [&](int t, int p) {  // sources 64 t + 1 + part + PARTS i of row rr of panel p
      const int r = row0 + p * PT + (int)rank * R + rr, src0 = row0 + t * PT + 1 + part;
      RowFactors<MODE, BWD, RC, PBC> f;
      f.load(w, min(r, N - 1));
#pragma unroll
      for (int i = 0; i < SRC; ++i) {
        fm[i] = (M_t)1.0;
        fe[i] = XZERO_E;
        if (r < N) f.h(w, src0 + PARTS * i, sm.T63, fm[i], fe[i]);
      }
    };
    int nt = 0, npan = first_panel(0);  // this warp's next task
    auto settle = [&] {
      while (nt < np && npan >= np) { ++nt; npan = first_panel(nt); }
    };
    settle();
    if (!RC && nt < np) load_factors(nt, npan);
    for (int t = 0; t + 2 < np; ++t) {
      int p = first_panel(t);
      if (p >= np) continue;
      handoff_wait(smem_addr(&sm.xbar[t]), 0, w.status, aborted);
      for (; p < np; p += S::BULK) {
        xi acc{sm.Am[p][lane], sm.Ae[p][lane]};
#pragma unroll
        for (int h = 0; h < SRC; h += 8) {
          xi y[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) y[i] = wire_get(&sm.X[t][part + PARTS * (h + i)]);
          if constexpr (RC) {
            const int r = row0 + p * PT + (int)rank * R + rr;
            RowFactors<MODE, BWD, true, PBC> f;
            f.load(w, min(r, N - 1));
            add_sources_rc<MODE, BWD, PBC, PARTS>(w, f, r < N, row0 + t * PT + 1 + part + PARTS * h, N - 1, y, sm.T63, acc);
          } else {
            unsigned long long kk[8];
            int e[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              kk[i] = mant53(fm[h + i]) << 11;
              e[i] = fe[h + i];
            }
            acc = xi_add(acc, xsum_fin<3>(xsum_dot<3, 8>(kk, e, y, 0, 2 * XZERO_E)));
          }
        }
        if (!RC) {
          npan += S::BULK;
          settle();
          if (nt < np) load_factors(nt, npan);
        }
        sm.Am[p][lane] = acc.m;
        sm.Ae[p][lane] = acc.e;
        if (p == t + 2) {
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_addr(&sm.done[p]));
        }
      }
    }
  } else if (!BWD && rank == 0) {
    // prefix sums C' of the superblock's rows
    double carry = t0 ? w.C[row0] : 0.0;
    long long ncarry = t0 ? *w.nsum : 0;
    for (int t = 2 * t0; t < 2 * (t0 + np) && t < w.NT; ++t) prefix_tile(w, t, carry, ncarry);
    if (lane == 0) {
      *w.nsum = ncarry;
      sm.misc[0] = carry;
      sm.nsum = ncarry;
    }
  }
  __syncwarp();
  cluster_arrive();
  if (!BWD && rank == 0 && (t0 + np) * PT >= N) {
    // V^{[1,N]} = C'[N] - (ln(y_N) - n ln 2)/beta and the normaliser 1/(N y_N)
    __syncthreads();
    const Wire &wy = sm.X[(N - 1 - row0) / PT][(N - 1) % PT];
    const xd yN = xi_to_xd(xi{wy.m, wy.e});
    if (tid == 0) {
      const xd inv = xnorm(1.0 / (yN.m * (double)N), -yN.e);
      w.scal[1] = inv.m;
      w.scal_i[0] = inv.e;
    } else if (tid == 32) {
      const double VB = reduced_potential(sm.misc[0], yN, sm.nsum, w.beta);
      w.scal[0] = VB;
      if (V_B) *V_B = VB;
      if (!isfinite(VB)) atomicOr(w.status, ST_NONFINITE);
    }
  }
  // No CTA leaves while a hand-off into its shared memory may be in flight:
  // each has waited for all of its own.  After an expired wait a hand-off may
  // still be on its way: give it time to land.
  cluster_wait();
  if (*(volatile int *)w.status & ST_TIMEOUT)
    for (int i = 0; i < 200; ++i) __nanosleep(1000);
}

// Cluster size CL (CTAs per recursion) is given at launch; blocks [0, CL) run
// the forward recursion, [CL, 2 CL) the backward one.
template <int MODE, int CL, bool RC>
__global__ void __launch_bounds__(ChainShape<CL>::THREADS, 1) chain_kernel(Workspace w, int t0, int np, double *V_B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ChainSmem &sm = *(ChainSmem *)smem_raw;
  // run_chain waits for the preceding grid (griddepcontrol.wait) once its
  // shared-memory set-up is done, before its first global-memory access
  if (RC && w.pbc) {
    if (blockIdx.x < CL) run_chain<MODE, false, CL, RC, RC>(w, t0, np, sm, V_B);
    else run_chain<MODE, true, CL, RC, RC>(w, t0, np, sm, V_B);
  } else {
    if (blockIdx.x < CL) run_chain<MODE, false, CL, RC, false>(w, t0, np, sm, V_B);
    else run_chain<MODE, true, CL, RC, false>(w, t0, np, sm, V_B);
  }
}

// ------------------------------------------------------ between superblocks
// Sources s0 .. s0+ns-1 (finished Y) added to the sums of the rows from r0 (a
// multiple of 32) on: one CTA per (row tile, recursion, slice of the sources),
// lane = row, a warp an eighth of the slice; the warps' sums meet in a fixed
// order.  `first`: the slice's sum starts here.  The next superblock's rows
// come first; the later ones are added while its recursions run (`beside`:
// launched behind them without waiting for them, as their predecessors' end
// was theirs to wait for; the first block waits before it ends, so that the
// next kernel's wait covers both).
constexpr int UPD_THREADS = 256, UPD_WARPS = UPD_THREADS / 32;
constexpr int UPD_MAX_SRC = 1024;  // sources of a slice staged at a time

template <int MODE, bool BWD, bool RC, bool PBC>
__device__ void source_update(const Workspace &w, int r0, int s0, int ns, bool first, Wire *Y,
                              const unsigned long long *T63, unsigned long long (*pm)[32], int (*pe)[32]) {
  using M_t = typename std::conditional<MODE == BPIMD_MIXED32, float, double>::type;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int r = r0 + blockIdx.x * TILE + lane, slice = blockIdx.z;
  const int per = (ns + SLICES - 1) / SLICES, lo = s0 + min(ns, slice * per), hi = s0 + min(ns, (slice + 1) * per);
  const double *gYm = BWD ? w.ybm : w.yfm;
  const int *gYe = BWD ? w.ybe : w.yfe;
  RowFactors<MODE, BWD, RC, PBC> f;
  f.load(w, min(r, w.N - 1));
  xi acc{1ull << 62, XZERO_E};
  for (int base = lo; base < hi; base += UPD_MAX_SRC) {
    const int n = min(UPD_MAX_SRC, hi - base), n8 = (n + 7) & ~7;
    __syncthreads();
    for (int i = threadIdx.x; i < n8; i += UPD_THREADS) {
      const xi y = i < n ? xi_from(xd{gYm[base + i], gYe[base + i]}) : xi{1ull << 62, XZERO_E};
      Y[i].m = y.m;
      Y[i].e = y.e;
    }
    __syncthreads();
    for (int i0 = 8 * wid; i0 < n8; i0 += 8 * UPD_WARPS) {
      xi y[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) y[i] = wire_get(&Y[i0 + i]);
      if constexpr (RC) {
        add_sources_rc<MODE, BWD, PBC, 1>(w, f, r < w.N, base + i0, base + n - 1, y, T63, acc);
      } else if (r < w.N) {
        unsigned long long kk[8];
        int e[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          M_t m;
          f.h(w, base + min(i0 + i, n - 1), T63, m, e[i]);
          kk[i] = mant53(m) << 11;
        }
        acc = xi_add(acc, xsum_fin<3>(xsum_dot<3, 8>(kk, e, y, 0, 2 * XZERO_E)));
      }
    }
  }
  pm[wid][lane] = acc.m;
  pe[wid][lane] = acc.e;
  __syncthreads();
  if (wid == 0 && r < w.N) {
    const size_t k = ((size_t)(BWD ? SLICES : 0) + slice) * w.N + r;
    if (!first) acc = xi_add(acc, xi{w.Asm[k], w.Ase[k]});
#pragma unroll
    for (int v = 1; v < UPD_WARPS; ++v) acc = xi_add(acc, xi{pm[v][lane], pe[v][lane]});
    w.Asm[k] = acc.m;
    w.Ase[k] = acc.e;
  }
}

template <int MODE, bool RC>
__global__ void __launch_bounds__(UPD_THREADS) source_update_kernel(Workspace w, int r0, int s0, int ns, bool first,
                                                                    bool beside) {
  __shared__ Wire Y[UPD_MAX_SRC];
  __shared__ unsigned long long pm[UPD_WARPS][32];
  __shared__ int pe[UPD_WARPS][32];
  __shared__ unsigned long long T63[RC ? 256 : 1];
  if (RC) pairg::table_init(T63);  // published by the staging's barrier
  if (!beside) {
    pdl_wait();
    pdl_trigger();
  }
  if (RC && w.pbc) {
    if (blockIdx.y == 0) source_update<MODE, false, RC, RC>(w, r0, s0, ns, first, Y, T63, pm, pe);
    else source_update<MODE, true, RC, RC>(w, r0, s0, ns, first, Y, T63, pm, pe);
  } else {
    if (blockIdx.y == 0) source_update<MODE, false, RC, false>(w, r0, s0, ns, first, Y, T63, pm, pe);
    else source_update<MODE, true, RC, false>(w, r0, s0, ns, first, Y, T63, pm, pe);
  }
  if (beside) {
    pdl_trigger();
    if (blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0) pdl_wait();
  }
}

constexpr int CHAIN_CLUSTER_LARGE = 16;

template <int MODE, int CL, bool RC>
cudaError_t launch_chain_cluster(const Workspace &w, double *V_B, cudaStream_t s) {
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = CL;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  const int panels = (w.N + PT - 1) / PT;
  cudaLaunchConfig_t cfg = {};
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.gridDim = dim3(4 * panels, 2);
  cfg.blockDim = dim3(PINV_THREADS);
  cfg.dynamicSmemBytes = sizeof(PinvSmem);
  cfg.numAttrs = 1;
  cudaError_t e = cudaLaunchKernelEx(&cfg, panel_inverse_kernel<MODE, RC>, w);
  const int sb = superblock_panels(panels, RC), rows = sb * PT;
  // superblock k's Y into the rows from r0 to r1
  auto update = [&](int k, int r0, int r1, bool beside) {
    const int s0 = k == 0 ? 0 : k * rows + 1, ns = (k + 1) * rows + 1 - s0;
    cfg.gridDim = dim3((r1 - r0 + TILE - 1) / TILE, 2, SLICES);
    cfg.blockDim = dim3(UPD_THREADS);
    cfg.dynamicSmemBytes = 0;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, source_update_kernel<MODE, RC>, w, r0, s0, ns, k == 0, beside);
  };
  for (int t0 = 0, k = 0; t0 < panels && e == cudaSuccess; t0 += sb, ++k) {
    const int np = panels - t0 < sb ? panels - t0 : sb, r0 = k * rows, r1 = r0 + rows;  // this superblock's rows
    if (k > 0) e = update(k - 1, r0, r1 < w.N ? r1 : w.N, false);
    if (e != cudaSuccess) return e;
    cfg.gridDim = dim3(2 * CL);
    cfg.blockDim = dim3(ChainShape<CL>::THREADS);
    cfg.dynamicSmemBytes = sizeof(ChainSmem);
    cfg.numAttrs = 2;
    e = cudaLaunchKernelEx(&cfg, chain_kernel<MODE, CL, RC>, w, t0, np, V_B);
    if (e == cudaSuccess && k > 0 && r1 < w.N) e = update(k - 1, r1, w.N, true);
  }
  return e;
}

// The kernel variant of a workspace: stored factors serve BPIMD_MIXED with the
// float64-layout code; the recompute mode has one variant per precision form.
template <int CL>
cudaError_t launch_chain_variant(const Workspace &w, double *V_B, cudaStream_t s) {
  if (!w.recomp)
    return w.mixed ? launch_chain_cluster<BPIMD_MIXED32, CL, false>(w, V_B, s)
                   : launch_chain_cluster<BPIMD_FP64, CL, false>(w, V_B, s);
  switch (w.mode) {
    case BPIMD_FP64: return launch_chain_cluster<BPIMD_FP64, CL, true>(w, V_B, s);
    case BPIMD_MIXED: return launch_chain_cluster<BPIMD_MIXED, CL, true>(w, V_B, s);
    default: return launch_chain_cluster<BPIMD_MIXED32, CL, true>(w, V_B, s);
  }
}

}  // namespace

// Once per process and device (host calls that must not sit between the
// launches of an evaluation): raise the dynamic shared-memory limit of the
// recursion kernels, allow the 16-CTA clusters, and check that two of them
// can be resident (else the 8-CTA form is used for every N).
namespace {
// per device: set up once under g_chain_mutex (two host threads making their
// first calls on one device must not both write these)
std::mutex g_chain_mutex;
bool g_chain_ready[64] = {false};
bool g_large_cluster[64] = {false};

template <int MODE, int CL, bool RC>
cudaError_t prepare_chain_kernel() {
  cudaError_t e = cudaFuncSetAttribute(chain_kernel<MODE, CL, RC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)sizeof(ChainSmem));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(panel_inverse_kernel<MODE, RC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(PinvSmem));
  if (e == cudaSuccess && CL > 8)
    e = cudaFuncSetAttribute(chain_kernel<MODE, CL, RC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}
template <int CL>
cudaError_t prepare_chain_variants() {
  cudaError_t e = prepare_chain_kernel<BPIMD_MIXED32, CL, false>();
  if (e == cudaSuccess) e = prepare_chain_kernel<BPIMD_FP64, CL, false>();
  if (e == cudaSuccess) e = prepare_chain_kernel<BPIMD_FP64, CL, true>();
  if (e == cudaSuccess) e = prepare_chain_kernel<BPIMD_MIXED, CL, true>();
  if (e == cudaSuccess) e = prepare_chain_kernel<BPIMD_MIXED32, CL, true>();
  return e;
}

template <int CL>
bool clusters_fit() {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * CL);
  cfg.blockDim = dim3(ChainShape<CL>::THREADS);
  cfg.dynamicSmemBytes = sizeof(ChainSmem);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  const bool ok =
      cudaOccupancyMaxActiveClusters(&n, chain_kernel<BPIMD_FP64, CL, true>, &cfg) == cudaSuccess && n >= 2;
  cudaGetLastError();
  return ok;
}
}  // namespace

cudaError_t prepare_chains() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_chain_mutex);
  if (g_chain_ready[dev]) return cudaSuccess;
  e = prepare_chains_small();
  if (e == cudaSuccess) e = prepare_chain_variants<CHAIN_CLUSTER>();
  if (e != cudaSuccess) return e;
  bool large = prepare_chain_variants<CHAIN_CLUSTER_LARGE>() == cudaSuccess;
  cudaGetLastError();
  large = large && clusters_fit<CHAIN_CLUSTER_LARGE>();
  g_large_cluster[dev] = large;
  g_chain_ready[dev] = true;
  return cudaSuccess;
}

cudaError_t launch_chains(const Workspace &w, double *V_B, cudaStream_t s) {
  if (!w.blocks) return cudaErrorInvalidValue;  // no panel-inverse storage in this workspace
  cudaError_t e = prepare_chains();
  if (e != cudaSuccess) return e;
  // One CTA per recursion with 32-row tiles and no panel inverses, against the
  // panels on clusters: N = 16 16.7 / 20.8 us, N = 64 20.5 / 25.5, N = 128
  // 25.5 / 26.6, N = 192 31.7 / 28.3.
  if (small_chain(w.N, w.mode) && !w.test_timeout) return launch_chains_small(w, V_B, s);
  int dev = 0;
  cudaGetDevice(&dev);
  bool large_ok;
  {
    std::lock_guard<std::mutex> lock(g_chain_mutex);
    large_ok = g_large_cluster[dev];
  }
  // 16 CTAs a recursion: N = 64 25.0 / 25.0 us (8 / 16 CTAs), N = 256 32.2 / 29.8,
  // N = 1024 82 / 60, N = 4096 536 / 390
  return large_ok ? launch_chain_variant<CHAIN_CLUSTER_LARGE>(w, V_B, s) : launch_chain_variant<CHAIN_CLUSTER>(w, V_B, s);
}

}  // namespace bpimd
