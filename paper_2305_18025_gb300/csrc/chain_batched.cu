// Forward and backward potential recursions of a batch of independent
// replicas (uneven N, P, beta): one CTA per recursion per replica, all in one
// launch.
//
// Same mathematics and the same dependent-step code as chain.cu (Eq.
// our-forward-potential-recurrence, Eq. backward-potential-recursion in linear
// space, tiles of 32 rows; see chain_common.cuh).  A small replica has little
// O(N^2) bulk per tile, so instead of a cluster per recursion every role sits
// in one CTA of 16 warps and many recursions share the GPU at once:
//   * warp 0: the 32 dependent steps of row tile t (chain_tile); then, once
//     they are done, warps 8..15 add its values to tile t+1's rows (four sources
//     each, from the staged off-diagonal block);
//   * warps off warp 0's sub-partition, numbered q = 0..11: q < 4 stage the
//     next diagonal block (8 rows each), q = 4, 5 the next off-diagonal block
//     (16 rows each), q = 6 forms the prefix sums (forward); all of them, once
//     that is done, add source tile t-1 to the row tiles >= t+1, one warp per
//     row tile, handed out by a counter;
//   * warps 4, 8, 12 share warp 0's sub-partition.  In a CTA that has an SM to
//     itself (single systems) they leave it to the chain, which sums on them
//     slowed from ~3100 to 6200-6800 cycles a tile; in a batch, where it is the
//     SM's throughput that counts, they take sums too.
// Y and the bulk row sums of the whole replica live in shared memory (32 bytes
// per particle), so N is bounded by BATCH_MAX_N.  Single systems of up to
// CHAIN_SMALL_N particles take the same code (launch_chains).  Tiles meet at
// __syncthreads.  CTAs are ordered by decreasing N (longest chains first).
#include <type_traits>

#include "chain_common.cuh"

namespace bpimd {
namespace {

using namespace chain_detail;

constexpr int BATCH_THREADS = 512;
constexpr int BATCH_COUPLE = 8;  // warps 8..15 couple a finished tile to the next

struct SingleSmem {
  unsigned long long Kdm[2 * BLK];
  double Hom[2 * BLK];  // MIXED: floats
  unsigned long long Pm[BATCH_COUPLE][TILE];  // the next tile's sums over this tile's values, by warp
  double misc[2];
  long long nsum;  // sum of the exponent parts n carried by y_N
  int Kde[2 * BLK];
  int Hoe[2 * BLK];
  int Pe[BATCH_COUPLE][TILE];
  int task[2];  // row tiles of the sums handed out, by parity of t
};

// Y (mantissa, xi mantissa, exponent) and the rows' sums (mantissa, exponent)
__host__ __device__ constexpr size_t single_smem_bytes(int N) {
  return sizeof(SingleSmem) + (size_t)(N + 1) * (2 * sizeof(double) + sizeof(int)) +
         (size_t)N * (sizeof(double) + sizeof(int));
}

// warp id -> role index q for warps off warp 0's sub-partition (-1 otherwise)
__device__ __forceinline__ int role_q(int wid) { return (wid & 3) ? wid - (wid >> 2) - 1 : -1; }

// MODE: BPIMD_MIXED32, or BPIMD_FP64 for both 64-bit forms (stored factors).
// ALONE: this CTA has its SM to itself (see above).
template <int MODE, bool BWD, bool ALONE>
__device__ void run_single(const Workspace &w, unsigned char *smem_raw, double *V_B) {
  constexpr bool MIXED = MODE == BPIMD_MIXED32;
  using M_t = typename std::conditional<MIXED, float, double>::type;
  const int N = w.N, NT = w.NT;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  SingleSmem &sm = *(SingleSmem *)smem_raw;
  double *Ym = (double *)(smem_raw + sizeof(SingleSmem));
  unsigned long long *Yk = (unsigned long long *)(Ym + (N + 1));
  unsigned long long *Am = Yk + (N + 1);  // MIXED32: float64 mantissas; else xi mantissas
  int *Ye = (int *)(Am + N);
  int *Ae = Ye + (N + 1);
  double *gYm = BWD ? w.ybm : w.yfm;
  int *gYe = BWD ? w.ybe : w.yfe;
  const int q = role_q(wid);

  for (int r = tid; r < N; r += blockDim.x) { Am[r] = MIXED ? 0ull : 1ull << 62; Ae[r] = XZERO_E; }
  if (tid == 0) { Ym[0] = 1.0; Yk[0] = 1ull << 62; Ye[0] = 0; gYm[0] = 1.0; gYe[0] = 0; }
  if (!BWD && tid == 0) w.C[0] = 0.0;
  if (tid < 2) sm.task[tid] = 0;
  if (q >= 0 && q < 4) stage_diag<MODE, BWD, 8>(w, 0, 8 * q, sm.Kdm, sm.Kde);
  if (q == 4 || q == 5) stage_offdiag<MODE, BWD, 16>(w, 0, 16 * (q - 4), sm.Hom, sm.Hoe);
  __syncthreads();

  xd cnext{1.0, 0};
  if (wid == 0 && lane < N) cnext = chain_coef<BWD>(w, lane);
  double carry = 0.0;
  long long ncarry = 0;
  for (int t = 0; t < NT; ++t) {
    const int buf = t & 1;
    if (wid == 0) {
      const int row = t * TILE + lane;
      const xd crow = cnext;
      if (row + TILE < N) cnext = chain_coef<BWD>(w, row + TILE);
      const int ra = min(row, N - 1);
      xi A;
      if constexpr (MIXED) A = xi_from(xd{__longlong_as_double((long long)Am[ra]), Ae[ra]});
      else A = xi{Am[ra], Ae[ra]};
      if (t >= 1) {  // the previous tile's values, in a fixed order
        int E = A.e;
#pragma unroll
        for (int k = 0; k < BATCH_COUPLE; ++k) E = max(E, sm.Pe[k][lane]);
        unsigned long long sum = A.m >> min(E - A.e + 4, 63);  // nine terms below 2^63: four bits of headroom
#pragma unroll
        for (int k = 0; k < BATCH_COUPLE; ++k) sum += sm.Pm[k][lane] >> min(E - sm.Pe[k][lane] + 4, 63);
        A = xsum_fin<4>(xsum{sum, E});
      }
      if (lane == 0) sm.task[buf ^ 1] = 0;
      chain_tile<MIXED>(N, t, A, crow, sm.Kdm + buf * BLK, sm.Kde + buf * BLK, Ym, Ye, Yk, gYm, gYe);
    } else if (q >= 0 || !ALONE) {
      if (q < 0) {
      } else if (q < 4) {
        if (t + 1 < NT)
          stage_diag<MODE, BWD, 8>(w, t + 1, 8 * q, sm.Kdm + (buf ^ 1) * BLK, sm.Kde + (buf ^ 1) * BLK);
      } else if (q < 6) {
        if (t + 1 < NT)
          stage_offdiag<MODE, BWD, 16>(w, t + 1, 16 * (q - 4), sm.Hom + (buf ^ 1) * BLK, sm.Hoe + (buf ^ 1) * BLK);
      } else if (q == 6) {
        if (!BWD) prefix_tile(w, t, carry, ncarry);
      }
      // source tile t-1 -> row tiles t+1.., one warp per row tile, taken as warps get free
      const int srcbase = (t - 1) * TILE;
      while (t >= 1) {
        int k = 0;
        if (lane == 0) k = atomicAdd(&sm.task[buf], 1);
        const int T = t + 1 + __shfl_sync(0xffffffffu, k, 0);
        if (T >= NT) break;
        const int r = T * TILE + lane;
        const int ra = r < N ? r : 0;
        RowFactors<MODE, BWD, false, false, 32> f;  // rows past N: their tile's padding (sums not kept)
        f.load(w, r);
        auto load = [&](int src, M_t &m, int &e) { f.h(w, src, nullptr, m, e); };
        if constexpr (MIXED) {
          float sacc = 0.0f;
          int E = XZERO_E;
#pragma unroll
          for (int h = 0; h < TILE; h += 16) {
            float m[16];
            int e[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              load(srcbase + h + i, m[i], e[i]);
            }
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const int v = srcbase + h + i;
              fmerge(sacc, E, mant_to_float(Ym[v]) * m[i], e[i] + Ye[v]);
            }
          }
          const xd acc = xnorm_int(xadd_int(xd{__longlong_as_double((long long)Am[ra]), Ae[ra]}, xd{f2d_int(sacc), E}));
          if (r < N) { Am[r] = (unsigned long long)__double_as_longlong(acc.m); Ae[r] = acc.e; }
        } else {
          // 64-bit integer products, as in chain.cu (a float64 FMA takes the
          // pipe ~75 cycles a warp: the 8 bulk warps waited for it)
          xi acc{Am[ra], Ae[ra]};
          double m[8];
          int e[8];
          if (ALONE)  // eight loads ahead; two CTAs on an SM hide them instead (and have fewer registers)
#pragma unroll
            for (int i = 0; i < 8; ++i) load(srcbase + i, m[i], e[i]);
#pragma unroll 1
          for (int h = 0; h < TILE; h += 8) {
            unsigned long long kk[8];
            int ke[8];
            xi y[8];
            if (!ALONE)
#pragma unroll
              for (int i = 0; i < 8; ++i) load(srcbase + h + i, m[i], e[i]);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              kk[i] = mant53(m[i]) << 11;
              ke[i] = e[i];
              y[i] = xi{Yk[srcbase + h + i], Ye[srcbase + h + i]};
            }
            if (ALONE && h + 8 < TILE)
#pragma unroll
              for (int i = 0; i < 8; ++i) load(srcbase + h + 8 + i, m[i], e[i]);
            acc = xi_add(acc, xsum_fin<3>(xsum_dot<3, 8>(kk, ke, y, 0, 2 * XZERO_E)));
          }
          if (r < N) { Am[r] = acc.m; Ae[r] = acc.e; }
        }
      }
    }
    __syncthreads();
    if (t + 1 < NT) {
      if (wid >= 8) {  // sources 32t + 4k .. +3 into tile t+1's rows
        const int k = wid - 8;
        const M_t *Hm = (const M_t *)(sm.Hom + buf * BLK);
        unsigned long long kk[4];
        int ke[4];
        xi y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int o = (4 * k + i) * 33 + lane, v = t * TILE + 4 * k + i;
          kk[i] = mant53(Hm[o]) << 11;
          ke[i] = sm.Hoe[buf * BLK + o];
          y[i] = xi{Yk[v], Ye[v]};
        }
        const xi p = xsum_fin<2>(xsum_dot<2, 4>(kk, ke, y, 0, 2 * XZERO_E));
        sm.Pm[k][lane] = p.m;
        sm.Pe[k][lane] = p.e;
      }
      __syncthreads();
    }
  }
  if (!BWD) {
    // V^{[1,N]} = C'[N] - (ln(y_N) - n ln 2)/beta, normaliser 1/(N y_N)
    if (q == 6 && lane == 0) { sm.misc[0] = carry; sm.nsum = ncarry; }
    __syncthreads();
    const xd yN{Ym[N], Ye[N]};
    if (tid == 0) {
      const xd inv = xnorm(1.0 / (yN.m * (double)N), -yN.e);
      w.scal[1] = inv.m;
      w.scal_i[0] = inv.e;
    }
    if (tid == 32) {
      const double VB = reduced_potential(sm.misc[0], yN, sm.nsum, w.beta);
      w.scal[0] = VB;
      if (V_B) *V_B = VB;
      if (!isfinite(VB)) atomicOr(w.status, ST_NONFINITE);
    }
  }
}

// A single small system of either 64-bit form: CTA d runs recursion d.
__global__ void __launch_bounds__(BATCH_THREADS) chain_small_kernel(Workspace w, double *V_B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  pdl_trigger();  // after the wait, never before it: what runs beside the recursions starts here without one
  if (blockIdx.x & 1) run_single<BPIMD_FP64, true, true>(w, smem_raw, nullptr);
  else run_single<BPIMD_FP64, false, true>(w, smem_raw, V_B);
}

// CTA 2k + d runs recursion d (0 forward, 1 backward) of replica order[k].
template <bool MIXED>
// Two CTAs per SM (64 registers a thread, no spills): each CTA's chain is
// latency-bound on one warp, so two replicas' recursions share an SM.
__global__ void __launch_bounds__(BATCH_THREADS, 2) chain_batched_kernel(const Workspace *__restrict__ ws,
                                                                         const int *__restrict__ order,
                                                                         double *V_B) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pdl_wait();
  pdl_trigger();  // after the wait, never before it: what runs beside the recursions starts here without one
  const int r = order[blockIdx.x >> 1];
  if (blockIdx.x & 1) run_single<MIXED ? BPIMD_MIXED32 : BPIMD_FP64, true, false>(ws[r], smem_raw, nullptr);
  else run_single<MIXED ? BPIMD_MIXED32 : BPIMD_FP64, false, false>(ws[r], smem_raw, V_B ? V_B + r : nullptr);
}

static_assert(single_smem_bytes(BATCH_MAX_N) <= 227 * 1024, "batched recursion state must fit in shared memory");
static_assert(BATCH_THREADS / 32 == 16, "role table assumes 16 warps");

}  // namespace

cudaError_t prepare_chains_small() {
  return cudaFuncSetAttribute(chain_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)single_smem_bytes(CHAIN_SMALL_N));
}

// BPIMD_FP64 and BPIMD_MIXED (BPIMD_MIXED32's chain has 32-bit words here, less
// than its single systems had)
cudaError_t launch_chains_small(const Workspace &w, double *V_B, cudaStream_t s) {
  return launch_pdl(chain_small_kernel, 2, BATCH_THREADS, single_smem_bytes(w.N), s, w, V_B);
}

cudaError_t launch_chains_batched(const Workspace *ws, const int *order, int R, int maxN, bool mixed, double *V_B,
                                  cudaStream_t s) {
  if (R <= 0) return cudaSuccess;
  static bool done[64] = {false};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && !done[dev]) {
    const int bytes = (int)single_smem_bytes(BATCH_MAX_N);
    e = cudaFuncSetAttribute(chain_batched_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(chain_batched_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
    done[dev] = true;
  }
  const size_t bytes = single_smem_bytes(maxN);
  e = mixed ? launch_pdl(chain_batched_kernel<true>, 2 * R, BATCH_THREADS, bytes, s, ws, order, V_B)
            : launch_pdl(chain_batched_kernel<false>, 2 * R, BATCH_THREADS, bytes, s, ws, order, V_B);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace bpimd
