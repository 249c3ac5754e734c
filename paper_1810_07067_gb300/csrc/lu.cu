// Batched LU with partial pivoting, complex128 and complex64, of matrices of one or of
// several orders (right-looking; one table entry a matrix, largest first).
//
// Two levels: panels of LU_NB columns inside outer blocks of LU_OB.  A panel is factored
// by a cluster of CTAs per matrix, its rows in shared memory (complex128,
// panel_cluster_kernel) or in registers (complex64, panel_reg_kernel); panel_kernel, one CTA
// in global memory, takes what no cluster holds.  Its interchanges and rows of U go to
// the rest of the outer block, which is updated; the block's interchanges, rows of U and
// one update of rank LU_OB then go to the columns right of it.  Updates are products on the
// tensor cores: exact digits for complex128 (lu_oz.cu), BF16 pieces for complex64 (R3
// below; its strips run on the CUDA cores).  Complex128 without a workspace updates the
// whole trailing matrix after every panel on the FP64 pipe.  Triangular solves: solve.cu.
#include <algorithm>
#include <array>
#include <cstdio>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include "smem.cuh"
#include "lu.cuh"
#include "lu_oz.cuh"

std::mutex& lu_capture_mutex() {
  static std::mutex m;
  return m;
}
#include "split3.cuh"
#include "tc.cuh"

namespace cg = cooperative_groups;

// Outer block of the complex64 factorization (see "two-level blocking" below).
#define LU_OB 128
#define LU_OB_CHUNKS (LU_OB / LU_NB)

// ---------------------------------------------------------------- panel
// Pivot measure: |a|^2 in FP64 for complex128; |Re a| + |Im a| in FP32 for
// complex64 (LAPACK's complex pivot measure; GB300's FP64 pipe is too slow to
// sit on the panel's critical path).  Largest measure, lowest row on ties.
// The FP64 measure is compared as an integer (the bits of a non-negative double
// keep its order; 0 = no candidate, NaN is never one): the comparisons of the
// search would otherwise queue on the FP64 pipe.
template <class T> struct Pivot;
template <> struct Pivot<cd> {
  using V = unsigned long long;
  static constexpr V NONE = 0, ZERO = 1;
  __device__ static V measure(cd a) {
    const V b = (V)__double_as_longlong(norm2(a));
    return b > 0x7FF0000000000000ull ? NONE : b + 1;
  }
  // 1 / a as conj(a) / |a|^2 with one division where |a|^2 is far from the ends of
  // the exponent range, by scaled division elsewhere
  __device__ static cd inverse(cd a) {
    const double q = norm2(a);
    const int e = (__double2hiint(q) >> 20) & 0x7FF;
    if (e < 64 || e > 1982) return cone<cd>() / a;
    const double r = 1.0 / q;
    return cd{a.x * r, -a.y * r};
  }
};
template <> struct Pivot<cf> {
  using V = float;
  static constexpr V NONE = -1.f, ZERO = 0.f;
  __device__ static V measure(cf a) { return fabsf(a.x) + fabsf(a.y); }
  __device__ static cf inverse(cf a) {
    const float q = fmaf(a.x, a.x, a.y * a.y);
    const int e = __float_as_int(q) >> 23;
    if (e < 32 || e > 222) return cone<cf>() / a;
    const float r = 1.f / q;
    return cf{a.x * r, -a.y * r};
  }
};

template <class V>
__device__ __forceinline__ void argmax_merge(V& v, int& idx, V v2, int i2) {
  if (v2 > v || (v2 == v && i2 < idx)) { v = v2; idx = i2; }
}

// The warp's largest measure and its lowest row, in every lane: redux on the words
// of an order-keeping integer instead of five rounds of shuffles.
__device__ __forceinline__ void warp_argmax(unsigned long long& v, int& idx) {
  const unsigned hi = (unsigned)(v >> 32), mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? (unsigned)v : 0u);
  const unsigned long long m = (unsigned long long)mh << 32 | ml;
  idx = (int)__reduce_min_sync(0xffffffffu, v == m ? (unsigned)idx : 0xffffffffu);
  v = m;
}
__device__ __forceinline__ void warp_argmax(float& v, int& idx) {
  // non-negative floats order as their bits; -1 (no candidate) and NaN, which is
  // never one, come out as 0 with the others' rows left out
  const unsigned b = v >= 0.f ? __float_as_uint(v) + 1u : 0u, m = __reduce_max_sync(0xffffffffu, b);
  idx = (int)__reduce_min_sync(0xffffffffu, b == m ? (unsigned)idx : 0xffffffffu);
  v = m ? __uint_as_float(m - 1u) : -1.f;
}

template <class T>
__global__ void __launch_bounds__(1024) panel_kernel(const LuMat* __restrict__ mats, int k0) {
  const LuMat mat = mats[blockIdx.x];
  const int n = mat.n;
  if (k0 >= n) return;
  const int nbk = min(LU_NB, n - k0);
  T* M = (T*)mat.A;
  int* pv = mat.piv;
  int* info = mat.info;
  using V = typename Pivot<T>::V;
  __shared__ V red_v[32];
  __shared__ int red_i[32];
  __shared__ int s_p;
  __shared__ T s_row[LU_NB];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5, NT = blockDim.x;
  for (int jj = 0; jj < nbk; ++jj) {
    const int c = k0 + jj;
    T* col = M + (size_t)c * n;
    V best = Pivot<T>::NONE;
    int bi = n;
    for (int r = c + tid; r < n; r += NT) argmax_merge(best, bi, Pivot<T>::measure(col[r]), r);
    for (int o = 16; o > 0; o >>= 1) {
      V v2 = __shfl_xor_sync(0xffffffffu, best, o);
      int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
      argmax_merge(best, bi, v2, i2);
    }
    if (lane == 0) { red_v[wid] = best; red_i[wid] = bi; }
    __syncthreads();
    if (wid == 0) {
      best = (lane < (NT >> 5)) ? red_v[lane] : Pivot<T>::NONE;
      bi = (lane < (NT >> 5)) ? red_i[lane] : n;
      for (int o = 16; o > 0; o >>= 1) {
        V v2 = __shfl_xor_sync(0xffffffffu, best, o);
        int i2 = __shfl_xor_sync(0xffffffffu, bi, o);
        argmax_merge(best, bi, v2, i2);
      }
      if (lane == 0) {
        s_p = (best > Pivot<T>::ZERO) ? bi : -1;
        pv[c] = (best > Pivot<T>::ZERO) ? bi : c;
        if (best <= Pivot<T>::ZERO && info[0] == 0) info[0] = c + 1;
      }
    }
    __syncthreads();
    const int p = s_p;
    if (p >= 0) {
      if (p != c && tid < nbk) {
        T* cc = M + (size_t)(k0 + tid) * n;
        T t = cc[c]; cc[c] = cc[p]; cc[p] = t;
      }
      __syncthreads();
      if (tid < nbk) s_row[tid] = M[(size_t)(k0 + tid) * n + c];
      __syncthreads();
      const T inv = cone<T>() / s_row[jj];
      for (int r = c + 1 + tid; r < n; r += NT) {
        T l = col[r] * inv;
        col[r] = l;
        // the row's remaining panel entries in chunks of 8: loads batched, then updates
        for (int c0 = jj + 1; c0 < nbk; c0 += 8) {
          T v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (c0 + u < nbk) v[u] = M[(size_t)(k0 + c0 + u) * n + r];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (c0 + u < nbk) M[(size_t)(k0 + c0 + u) * n + r] = v[u] - l * s_row[c0 + u];
        }
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- cluster panel
// The panel (rows k0..n-1, nbk columns) held in the shared memory of a
// cluster of C CTAs: CTA q owns rows k0 + q R .. k0 + (q+1) R - 1 as a
// column-major slice [nbk][R].  Per column: every CTA writes its candidate
// (value, row index, reciprocal and the row itself) into every CTA's shared
// memory through the cluster's distributed shared memory, and CTA 0, which owns
// row c whenever C > 1 (then R > LU_NB), writes row c as well; one cluster
// barrier; every CTA picks the winner, the pivot's owner takes row c, CTA 0 takes
// the pivot row; the multipliers are formed and applied to the next column alone,
// which is searched in the same pass. The update of the columns behind it runs
// between the arrival at the next column's cluster barrier and the wait there; the
// two rows that travel are brought up to date by the warps that send them. A column
// is a chain of some twenty dependent FP64 operations, two reductions and the
// exchange, and the rank-1 update, bound by the FP64 pipe, now runs beside the
// reciprocal and the exchange instead of after them. A dependent FP64 operation
// takes 65 clocks and an SM issues one for a warp every 19, so the update goes over
// (column, row) pairs without idle lanes. One column of a 1250-row panel in eight
// CTAs: 6.5 -> 4.4 us; factorization of 9 matrices of order 1250: 16.7 -> 13.9 ms.
// Same pivot rule as panel_kernel (largest |a|^2, lowest row on ties), and every
// element takes the same updates in the same order.
#define PANEL_SMEM_MAX (200 * 1024)
#define PANEL_THREADS 512

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }

template <class T>
__global__ void __launch_bounds__(PANEL_THREADS) panel_cluster_kernel(const LuMat* __restrict__ mats, int k0, int R) {
  cg::cluster_group cl = cg::this_cluster();
  const int C = (int)cl.num_blocks();
  const int q = (int)cl.block_rank();
  const LuMat mat = mats[blockIdx.y];  // the whole cluster works on one matrix
  const int n = mat.n;
  if (k0 >= n) return;                 // every CTA of the cluster, before any cluster barrier
  const int nbk = min(LU_NB, n - k0);
  T* M = (T*)mat.A;
  int* pv = mat.piv;
  int* info = mat.info;
  extern __shared__ __align__(16) unsigned char panel_smem[];
  T* a = (T*)panel_smem;  // [nbk][R]
  using V = typename Pivot<T>::V;
  // exchange slots, three deep: a CTA reads the pivot row of column jj until it
  // arrives at the cluster barrier of column jj + 2, which every peer passes before
  // it writes the slot again for column jj + 3
  __shared__ V cand_v[3][8];
  __shared__ int cand_i[3][8];
  __shared__ T cand_row[3][8][LU_NB];   // each CTA's candidate row of the panel
  __shared__ T cand_inv[3][8];          // and the reciprocal of its candidate
  __shared__ T top_row[3][LU_NB];       // row c (CTA 0 owns every row c of the panel)
  __shared__ V red_v[PANEL_THREADS / 32];
  __shared__ int red_i[PANEL_THREADS / 32];
  __shared__ int s_bi;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int row0 = k0 + q * R;
  const int nr = max(0, min(R, n - row0));  // rows owned by this CTA
  for (int t = tid; t < nbk * nr; t += PANEL_THREADS) {
    int r = t % nr, j = t / nr;
    a[j * R + r] = M[(size_t)(k0 + j) * n + row0 + r];
  }
  cl.sync();  // every CTA of the cluster has started before a peer writes to its shared memory
  V best = Pivot<T>::NONE;
  int bi = n;
  for (int r = tid; r < nr; r += PANEL_THREADS) argmax_merge(best, bi, Pivot<T>::measure(a[r]), row0 + r);
  warp_argmax(best, bi);
  if (lane == 0) { red_v[wid] = best; red_i[wid] = bi; }
  T trav = czero<T>();
  const T* pend = nullptr;  // pivot row of column jj - 1 while its update of columns jj + 1.. is due
  for (int jj = 0, buf = 0; jj < nbk; ++jj, buf = buf == 2 ? 0 : buf + 1) {
    const int c = k0 + jj;
    const T* aj = a + jj * R;
    __syncthreads();
    if (wid == 0) {
      best = (lane < PANEL_THREADS / 32) ? red_v[lane] : Pivot<T>::NONE;
      bi = (lane < PANEL_THREADS / 32) ? red_i[lane] : n;
      warp_argmax(best, bi);
      if (lane == 0) s_bi = bi;
    }
    __syncthreads();
    const int rb = s_bi < n ? s_bi - row0 : -1, rc = q == 0 ? c - row0 : -1;  // rows that travel
    if (wid == 0) {
      if (lane < C) {  // this CTA's candidate into slot q of every CTA
        cl.map_shared_rank(cand_v[buf], lane)[q] = best;
        cl.map_shared_rank(cand_i[buf], lane)[q] = bi;
        cl.map_shared_rank(cand_inv[buf], lane)[q] = rb >= 0 ? Pivot<T>::inverse(aj[rb]) : czero<T>();
      }
    } else if (wid < 3 && lane < nbk) {
      // the candidate row (warp 1) and row c (warp 2), brought up to date, into every
      // CTA; where they are the same row warp 1 alone keeps the updated values
      const int r = wid == 1 ? rb : rc;
      if (r >= 0) {
        T v = a[lane * R + r];
        if (pend && lane > jj) {
          const T l = a[(jj - 1) * R + r];
          v = v - l * pend[lane];
        }
        for (int u = 0; u < C; ++u) cl.map_shared_rank(wid == 1 ? cand_row[buf][q] : top_row[buf], u)[lane] = v;
        trav = v;
      }
    }
    cluster_arrive();
    if (pend) {  // the other rows, as one list of (column, row): no lane of the FP64 pipe idles
      const int r0 = max(0, c - row0), nrow = nr - r0, j0 = jj + 1;
      int t = PANEL_THREADS - 1 - tid;  // warps 0..2, busy above, take the list's end
      if (nrow > 0) {
        const int sj = PANEL_THREADS / nrow, sr = PANEL_THREADS - sj * nrow;
        int j = t / nrow, r = t - j * nrow;
        for (j += j0, r += r0; j < nbk;) {
          if (r != rb && r != rc) a[j * R + r] = a[j * R + r] - a[(jj - 1) * R + r] * pend[j];
          j += sj;
          r += sr;
          if (r >= nr) { r -= nrow; ++j; }
        }
      }
    }
    cluster_wait();
    if (pend && lane > jj && lane < nbk && (wid == 1 || (wid == 2 && rc != rb)) && (wid == 1 ? rb : rc) >= 0)
      a[lane * R + (wid == 1 ? rb : rc)] = trav;
    __syncthreads();
    best = Pivot<T>::NONE;
    bi = n;
    int win = -1;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const V v2 = cand_v[buf][u];  // slots from C on are read and passed over
      const int i2 = cand_i[buf][u];
      if (u < C && (v2 > best || (v2 == best && i2 < bi))) { best = v2; bi = i2; win = u; }
    }
    const int p = (best > Pivot<T>::ZERO) ? bi : -1;
    if (q == 0 && tid == 0) {
      pv[c] = (p >= 0) ? p : c;
      if (p < 0 && info[0] == 0) info[0] = c + 1;
    }
    const int jn = jj + 1;  // the next column, searched as it is updated
    const T* prow = cand_row[buf][p >= 0 ? win : 0];
    const T* trow = top_row[buf];
    if (p >= 0 && wid == PANEL_THREADS / 32 - 1 && lane < nbk) {
      // row c moves to p (columns jj and jn there are formed below), the pivot row to c
      if (p != c && q == (p - k0) / R && lane != jj && lane != jn) a[lane * R + p - row0] = trow[lane];
      if (q == 0) a[lane * R + c - row0] = prow[lane];
    }
    best = Pivot<T>::NONE;
    bi = n;
    if (p >= 0) {
      const T inv = cand_inv[buf][win];
      const T pn = jn < nbk ? prow[jn] : czero<T>();
      for (int r = max(0, c + 1 - row0) + tid; r < nr; r += PANEL_THREADS) {
        const bool sw = row0 + r == p;
        const T l = (sw ? trow[jj] : a[jj * R + r]) * inv;
        a[jj * R + r] = l;
        if (jn < nbk) {
          const T v = (sw ? trow[jn] : a[jn * R + r]) - l * pn;
          a[jn * R + r] = v;
          argmax_merge(best, bi, Pivot<T>::measure(v), row0 + r);
        }
      }
    } else if (jn < nbk) {
      for (int r = max(0, c + 1 - row0) + tid; r < nr; r += PANEL_THREADS)
        argmax_merge(best, bi, Pivot<T>::measure(a[jn * R + r]), row0 + r);
    }
    pend = p >= 0 ? prow : nullptr;
    warp_argmax(best, bi);
    if (lane == 0) { red_v[wid] = best; red_i[wid] = bi; }
  }
  __syncthreads();
  for (int t = tid; t < nbk * nr; t += PANEL_THREADS) {
    int r = t % nr, j = t / nr;
    M[(size_t)(k0 + j) * n + row0 + r] = a[j * R + r];
  }
  cl.sync();  // no CTA leaves while a peer could still address its shared memory
}

static int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms <= 0) {
    cudaGetLastError();
    sms = 1;
  }
  return sms;
}

// Cluster size: of the sizes 1..8 whose row slices of the largest matrix (rows =
// its n - k0) fit the shared memory, the one whose estimated time for the batch is
// least.  A column costs a chain of about 6000 clocks and 61 clocks for each of its
// CTA's rows, times the CTAs that share an SM (the FP64 pipe bounds the updates);
// clusters stay within a group of SMs, so a batch that fills the device takes whole
// waves, and the sizes that are no power of two often need one wave less (65
// matrices of order 1280: 3 waves of 32 clusters of eight, 2 of 40 of seven;
// 48.4 -> 47.7 ms; 9 of order 1250 with eight CTAs instead of two: 15.2 -> 13.7 ms).
// Smaller matrices of a ragged batch own fewer rows of the same slices.
// Returns false (nothing launched) when none fits or no such cluster can be
// resident; the caller then uses panel_kernel.
template <class T>
static bool launch_panel_cluster(const LuMat* mats, int rows, int k0, int batch, cudaStream_t s) {
  static bool attr = false;
  if (!attr) {
    if (cudaFuncSetAttribute(panel_cluster_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, PANEL_SMEM_MAX) !=
        cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    attr = true;
  }
  const int sms = sm_count();
  cudaLaunchAttribute at[1];
  cudaLaunchConfig_t best = {};
  int bestR = 0;
  double cost = 0.0;
  for (int C = 1; C <= 8; ++C) {
    const int R = (rows + C - 1) / C;
    const size_t smem = (size_t)LU_NB * R * sizeof(T);
    if (smem > PANEL_SMEM_MAX || (C > 1 && R <= LU_NB)) continue;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(C, batch);
    cfg.blockDim = dim3(PANEL_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, panel_cluster_kernel<T>, &cfg) != cudaSuccess || ncl < 1) {
      cudaGetLastError();
      continue;
    }
    const int waves = (batch + ncl - 1) / ncl, share = (std::min(batch, ncl) * C + sms - 1) / sms;
    const double t = waves * (6000.0 + 61.0 * R * share);
    if (!bestR || t < cost) {
      cost = t;
      best = cfg;
      bestR = R;
    }
  }
  if (!bestR) return false;
  at[0].val.clusterDim.x = best.gridDim.x;
  if (cudaLaunchKernelEx(&best, panel_cluster_kernel<T>, mats, k0, bestR) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

// ---------------------------------------------------------------- register panel
// Complex64 panel with the rows in registers: CTA q of a cluster of C owns
// rows k0 + q R .. k0 + (q+1) R - 1 (R = PREG_THREADS x PREG_RPT), thread t
// rows t + PREG_THREADS s (s < PREG_RPT), all LU_NB columns of each (the
// column loop is unrolled, so every register index is static).  Per column:
// local argmax (warp shuffles, then across the CTA's warps); the candidate
// row is staged in shared memory by its owner (and row c by its owner in CTA
// 0, which holds the panel's first R > LU_NB rows); every CTA's candidate
// (value, index, row) and row c reach every CTA through distributed shared
// memory (slots double-buffered by column parity); one cluster barrier; then
// each thread applies the interchange and the rank-1 update to its own rows.
// Same pivot rule and arithmetic as panel_cluster_kernel.
#define PREG_THREADS 256
#define PREG_RPT 2
#define PREG_R (PREG_THREADS * PREG_RPT)

struct PregShared {
  float cand_v[2][8];
  int cand_i[2][8];
  cf cand_row[2][8][LU_NB];  // each CTA's candidate row
  cf top_row[2][LU_NB];      // row c
  cf loc_row[LU_NB], loc_top[LU_NB];
  float red_v[PREG_THREADS / 32];
  int red_i[PREG_THREADS / 32];
};
struct PregCtx {
  int k0, n, nbk, C, q, tid, lane, wid;
  int* pv;
  int* info;
};

// Column jj of the panel.  The column loop is not unrolled (a fully unrolled
// panel overflows the instruction cache); every register access uses a
// compile-time column index, the column jj itself being picked out by a select
// over the 8 columns of its eighth-aligned group, and the rank-1 update skips the
// groups left of it and has no predicates right of it.  What bounds it is the
// chain of a column: at 4096 rows in eight CTAs 5700 -> 4200 clocks of select 350,
// search 450, staging and exchange 1700, exchange of rows 350, update 1070 (65
// matrices of order 1280: 14.8 -> 12.8 ms; 5 of order 2048: 12.0 -> 9.2 ms).
__device__ __forceinline__ void preg_column(int jj, const cg::cluster_group& cl, PregShared& sh, const PregCtx& x,
                                            cf (&a)[PREG_RPT][LU_NB], const int (&grow)[PREG_RPT]) {
  const int c = x.k0 + jj, buf = jj & 1, n = x.n;
  cf colv[PREG_RPT];
#pragma unroll
  for (int g = 0; g < LU_NB; g += 8)
    if (jj >= g && jj < g + 8) {
#pragma unroll
      for (int s = 0; s < PREG_RPT; ++s) {
        cf t[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) t[j] = jj & 4 ? a[s][g + 4 + j] : a[s][g + j];
        t[0] = jj & 2 ? t[2] : t[0];
        t[1] = jj & 2 ? t[3] : t[1];
        colv[s] = jj & 1 ? t[1] : t[0];
      }
    }
  float best = -1.f;
  int bi = n;
#pragma unroll
  for (int s = 0; s < PREG_RPT; ++s)
    if (grow[s] >= c && grow[s] < n) argmax_merge(best, bi, Pivot<cf>::measure(colv[s]), grow[s]);
  warp_argmax(best, bi);
  if (x.lane == 0) { sh.red_v[x.wid] = best; sh.red_i[x.wid] = bi; }
  __syncthreads();
  best = x.lane < PREG_THREADS / 32 ? sh.red_v[x.lane] : -1.f;
  bi = x.lane < PREG_THREADS / 32 ? sh.red_i[x.lane] : n;
  warp_argmax(best, bi);
#pragma unroll
  for (int s = 0; s < PREG_RPT; ++s) {
    if (grow[s] == bi) {
#pragma unroll
      for (int j = 0; j < LU_NB; ++j) sh.loc_row[j] = a[s][j];
    }
    if (x.q == 0 && grow[s] == c) {
#pragma unroll
      for (int j = 0; j < LU_NB; ++j) sh.loc_top[j] = a[s][j];
    }
  }
  __syncthreads();
  if (x.tid < 32 * x.C) {
    const int j = x.tid & 31, u = x.tid >> 5;
    if (j < x.nbk) {
      if (bi < n) cl.map_shared_rank(&sh.cand_row[buf][x.q][0], u)[j] = sh.loc_row[j];
      if (x.q == 0) cl.map_shared_rank(&sh.top_row[buf][0], u)[j] = sh.loc_top[j];
    }
    if (j == 0) {
      cl.map_shared_rank(&sh.cand_v[buf][0], u)[x.q] = best;
      cl.map_shared_rank(&sh.cand_i[buf][0], u)[x.q] = bi;
    }
  }
  if (x.C > 1) cl.sync();
  else __syncthreads();
  float bv = x.lane < x.C ? sh.cand_v[buf][x.lane] : -1.f;
  int p = x.lane < x.C ? sh.cand_i[buf][x.lane] : n;
  const int own = p;
  warp_argmax(bv, p);
  const int win = max(0, __ffs(__ballot_sync(0xffffffffu, own == p && x.lane < x.C)) - 1);
  const bool ok = bv > 0.f;
  if (x.q == 0 && x.tid == 0) {
    x.pv[c] = ok ? p : c;
    if (!ok && x.info[0] == 0) x.info[0] = c + 1;
  }
  if (!ok) return;
  const cf* prow = sh.cand_row[buf][win];
  const cf* trow = sh.top_row[buf];
#pragma unroll
  for (int s = 0; s < PREG_RPT; ++s) {
    if (grow[s] == c) {  // row c takes the pivot row
#pragma unroll
      for (int j = 0; j < LU_NB; ++j) a[s][j] = prow[j];
    } else if (grow[s] == p) {  // the pivot's row takes row c
#pragma unroll
      for (int j = 0; j < LU_NB; ++j) a[s][j] = trow[j];
      colv[s] = trow[jj];
    }
  }
  const cf inv = Pivot<cf>::inverse(prow[jj]);
  cf l[PREG_RPT];
  bool act[PREG_RPT];
#pragma unroll
  for (int s = 0; s < PREG_RPT; ++s) {
    l[s] = colv[s] * inv;
    act[s] = grow[s] > c && grow[s] < n;
  }
#pragma unroll
  for (int g = 0; g < LU_NB; g += 8) {
    if (jj >= g + 8) continue;
    cf u[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) u[j] = prow[g + j];
    if (jj < g) {
#pragma unroll
      for (int s = 0; s < PREG_RPT; ++s)
        if (act[s]) {
#pragma unroll
          for (int j = 0; j < 8; ++j) a[s][g + j] = a[s][g + j] - l[s] * u[j];
        }
    } else {
#pragma unroll
      for (int s = 0; s < PREG_RPT; ++s)
        if (act[s]) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (g + j > jj) a[s][g + j] = a[s][g + j] - l[s] * u[j];
            else if (g + j == jj) a[s][g + j] = l[s];
          }
        }
    }
  }
}

__global__ void __launch_bounds__(PREG_THREADS, 1) panel_reg_kernel(const LuMat* __restrict__ mats, int k0) {
  cg::cluster_group cl = cg::this_cluster();
  const LuMat mat = mats[blockIdx.y];  // the whole cluster works on one matrix
  const int n = mat.n;
  if (k0 >= n) return;                 // every CTA of the cluster, before any cluster barrier
  __shared__ PregShared sh;
  PregCtx x;
  x.k0 = k0;
  x.n = n;
  x.nbk = min(LU_NB, n - k0);
  x.C = (int)cl.num_blocks();
  x.q = (int)cl.block_rank();
  x.tid = threadIdx.x;
  x.lane = threadIdx.x & 31;
  x.wid = threadIdx.x >> 5;
  x.pv = mat.piv;
  x.info = mat.info;
  cf* M = (cf*)mat.A;
  const int row0 = k0 + x.q * PREG_R;
  int grow[PREG_RPT];
  cf a[PREG_RPT][LU_NB];
#pragma unroll
  for (int s = 0; s < PREG_RPT; ++s) {
    grow[s] = row0 + x.tid + PREG_THREADS * s;
#pragma unroll
    for (int j = 0; j < LU_NB; ++j)
      a[s][j] = (grow[s] < n && j < x.nbk) ? M[(size_t)(k0 + j) * n + grow[s]] : CF(0.f);
  }
#pragma unroll 1
  for (int jj = 0; jj < x.nbk; ++jj) preg_column(jj, cl, sh, x, a, grow);
#pragma unroll
  for (int s = 0; s < PREG_RPT; ++s)
    if (grow[s] < n) {
#pragma unroll
      for (int j = 0; j < LU_NB; ++j)
        if (j < x.nbk) M[(size_t)(k0 + j) * n + grow[s]] = a[s][j];
    }
  cl.sync();  // no CTA leaves while a peer could still address its shared memory
}

// Cluster of C = ceil(rows / PREG_R) <= 8 CTAs; false when the panel is taller
// or no such cluster can be resident.
static bool launch_panel_reg(const LuMat* mats, int rows, int k0, int batch, cudaStream_t s) {
  const int C = (rows + PREG_R - 1) / PREG_R;
  if (C < 1 || C > 8) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(C, batch);
  cfg.blockDim = dim3(PREG_THREADS);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = C;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int nclusters = 0;
  if (cudaOccupancyMaxActiveClusters(&nclusters, panel_reg_kernel, &cfg) != cudaSuccess || nclusters < 1) {
    cudaGetLastError();
    return false;
  }
  if (cudaLaunchKernelEx(&cfg, panel_reg_kernel, mats, k0) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return true;
}

// ---------------------------------------------------------------- swaps
// The nbk interchanges of a block column compose to a permutation of at most
// 2 nbk rows: the block's own rows (slots 0..nbk-1) and the distinct targets
// below it (slot nbk + lane of the first interchange naming it).  One warp
// forms it per CTA; each warp then moves the affected entries of its columns
// (all loads before all stores).
//
// Columns (mode): 0 all but the panel's own; 1 those left of the panel and
// the rest of its LU_OB block (columns < min(K0 + LU_OB, n)); 2 those right
// of the block.
#define SWAP_COLS 64
template <class T>
__global__ void __launch_bounds__(256) swap_kernel(const LuMat* __restrict__ mats, int k0, int K0, int mode) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n;
  if (k0 >= n) return;
  const int nbk = min(LU_NB, n - k0);
  const int bend = min(K0 + LU_OB, n);
  const int lo = mode == 2 ? bend : 0, hi = mode == 1 ? bend : n;
  const bool skip = mode != 2;  // the panel's columns lie inside [lo, hi)
  const int ncols = hi - lo - (skip ? nbk : 0);
  const int* piv = mat.piv;
  __shared__ int pos[2 * LU_NB], src[2 * LU_NB], slot[LU_NB];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kend = k0 + nbk;
  if (warp == 0) {
    const int p = (lane < nbk) ? piv[k0 + lane] : -1;
    const unsigned same = __match_any_sync(0xffffffffu, p);
    const bool below = p >= kend;
    const bool first = below && (__ffs(same) - 1 == lane);
    const int sp = (lane >= nbk) ? 0 : (below ? LU_NB + __ffs(same) - 1 : p - k0);
    pos[lane] = (lane < nbk) ? k0 + lane : -1;
    src[lane] = pos[lane];
    pos[LU_NB + lane] = first ? p : -1;
    src[LU_NB + lane] = first ? p : -1;
    slot[lane] = sp;
    __syncwarp();
    if (lane == 0)
      for (int k = 0; k < nbk; ++k) {
        const int s2 = slot[k];
        if (s2 != k) { int t = src[k]; src[k] = src[s2]; src[s2] = t; }
      }
  }
  __syncthreads();
  const int d0 = pos[lane], d1 = pos[lane + 32], s0 = src[lane], s1 = src[lane + 32];
  for (int cc = warp; cc < SWAP_COLS; cc += 8) {
    const int idx = blockIdx.x * SWAP_COLS + cc;
    if (idx >= ncols) break;  // whole warp
    int c = lo + idx;
    if (skip && c >= k0) c += nbk;  // skip the panel's own columns
    T* col = (T*)mat.A + (size_t)c * n;
    T v0 = czero<T>(), v1 = czero<T>();
    if (d0 >= 0 && d0 != s0) v0 = col[s0];
    if (d1 >= 0 && d1 != s1) v1 = col[s1];
    __syncwarp();
    if (d0 >= 0 && d0 != s0) col[d0] = v0;
    if (d1 >= 0 && d1 != s1) col[d1] = v1;
    __syncwarp();
  }
}

// ---------------------------------------------------------------- U12 = L11^{-1} A12
// Complex128 without a workspace: all columns right of the panel, one thread a column.
__global__ void trsm_kernel(const LuMat* __restrict__ mats, int k0) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n;
  if (k0 + LU_NB >= n) return;  // no columns right of the panel (or the panel is the last)
  cd* M = (cd*)mat.A;
  __shared__ cd L[LU_NB][LU_NB + 1];
  for (int t = threadIdx.x; t < LU_NB * LU_NB; t += blockDim.x) {
    const int r = t % LU_NB, cc = t / LU_NB;
    L[r][cc] = M[(size_t)(k0 + cc) * n + k0 + r];
  }
  __syncthreads();
  const int c = k0 + LU_NB + blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= n) return;
  cd* col = M + (size_t)c * n + k0;
  cd x[LU_NB];
#pragma unroll
  for (int r = 0; r < LU_NB; ++r) x[r] = col[r];
#pragma unroll
  for (int k = 0; k < LU_NB; ++k) {
#pragma unroll
    for (int r = k + 1; r < LU_NB; ++r) x[r] = x[r] - L[r][k] * x[k];
  }
#pragma unroll
  for (int r = 0; r < LU_NB; ++r) col[r] = x[r];
}

// The same for complex64, one thread a column: the rows of 128 columns pass through
// shared memory, a warp to a column, so that they are read and written whole (a
// thread walking its own column in memory waited for it: N = 1024, 129 modes,
// 19.1 -> 8.4 ms).
__global__ void __launch_bounds__(128) trsm_c64_kernel(const LuMat* __restrict__ mats, int k0, int K0, int mode) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n;
  if (k0 + LU_NB >= n) return;  // no columns right of the panel (or the panel is the last)
  const int c0 = mode == 2 ? K0 + LU_OB : k0 + LU_NB, c1 = mode == 1 ? min(K0 + LU_OB, n) : n;
  const int j0 = c0 + blockIdx.x * 128, nc = min(128, c1 - j0);
  if (nc <= 0) return;
  cf* M = (cf*)mat.A;
  __shared__ cf L[LU_NB][LU_NB + 1];
  __shared__ cf X[128][LU_NB + 1];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int c = warp; c < LU_NB; c += 4) L[lane][c] = M[(size_t)(k0 + c) * n + k0 + lane];
#pragma unroll 8
  for (int c = warp; c < nc; c += 4) X[c][lane] = M[(size_t)(j0 + c) * n + k0 + lane];
  __syncthreads();
  if (tid < nc) {
    cf x[LU_NB];
#pragma unroll
    for (int r = 0; r < LU_NB; ++r) x[r] = X[tid][r];
#pragma unroll
    for (int k = 0; k < LU_NB; ++k)
#pragma unroll
      for (int r = k + 1; r < LU_NB; ++r) x[r] = x[r] - L[r][k] * x[k];
#pragma unroll
    for (int r = 0; r < LU_NB; ++r) X[tid][r] = x[r];
  }
  __syncthreads();
#pragma unroll 8
  for (int c = warp; c < nc; c += 4) M[(size_t)(j0 + c) * n + k0 + lane] = X[c][lane];
}

// ---------------------------------------------------------------- trailing update
// Complex128 without a workspace, on the FP64 pipe:
// C[i0.., j0..] -= A[i0.., k0..k0+nbk) * A[k0..k0+nbk), j0..], 64x64 tiles,
// 256 threads, each 4x4 outputs: rows tx + 16a, columns ty + 16b.
#define GT 64
__global__ void __launch_bounds__(256) gemm_update_kernel(const LuMat* __restrict__ mats, int k0) {
  const LuMat mat = mats[blockIdx.z];
  const int n = mat.n;
  const int nbk = LU_NB;
  const int start = k0 + nbk;
  if ((int)blockIdx.x * GT >= n - start || (int)blockIdx.y * GT >= n - start) return;
  cd* M = (cd*)mat.A;
  const int i0 = start + blockIdx.x * GT, j0 = start + blockIdx.y * GT;
  __shared__ cd As[LU_NB][GT];
  __shared__ cd Bs[LU_NB][GT];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  for (int t = tid; t < nbk * GT; t += 256) {
    int r = t % GT, kk = t / GT;
    int gi = i0 + r;
    As[kk][r] = (gi < n) ? M[(size_t)(k0 + kk) * n + gi] : C(0.0);
    int kb = t % nbk, cj = t / nbk;  // B element (row k0+kb, column j0+cj)
    int gj = j0 + cj;
    Bs[kb][cj] = (gj < n) ? M[(size_t)gj * n + k0 + kb] : C(0.0);
  }
  __syncthreads();
  cd acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[a][c] = C(0.0);
  for (int kk = 0; kk < nbk; ++kk) {
    cd av[4], bv[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) av[a] = As[kk][tx + 16 * a];
#pragma unroll
    for (int c = 0; c < 4; ++c) bv[c] = Bs[kk][ty + 16 * c];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][c] = fma(av[a], bv[c], acc[a][c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    int gj = j0 + ty + 16 * c;
    if (gj >= n) continue;
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      int gi = i0 + tx + 16 * a;
      if (gi < n) {
        cd* d = M + (size_t)gj * n + gi;
        *d = *d - acc[a][c];
      }
    }
  }
}

// ---------------------------------------------------------------- two-level blocking (complex64)
// The complex64 factorization works on outer blocks of LU_OB = 4 LU_NB
// columns.  Inside a block, each LU_NB panel is factored, its interchanges
// are applied to the columns left of it and to the rest of the block, its
// rows of U are formed within the block, and the block's remaining columns
// are updated (all rows below: "R1").  Then the columns right of the block
// take the block's interchanges, in order, and the block's rows of U there
// are formed panel by panel (each panel's triangular solve followed by the
// update of the block's remaining rows: "R2").  Last, the trailing matrix
// right of and below the block ("R3") receives the four panels' updates
// together, as one rank-LU_OB product on the tensor cores, so it is read and
// written once per LU_OB columns instead of once per LU_NB.  (The columns
// right of the block must not take a panel's interchanges before the block
// is done: a row from below the block, without the deferred updates, would
// trade places with a row inside it, with them.)

// Strip update on the CUDA cores (FP32 arithmetic): C -= L U with
// L = A[r0..r1, k..k+LU_NB), U = A[k..k+LU_NB, c0..c1); which = 1 gives the
// block-column strip (rows k+LU_NB..n, columns k+LU_NB..min(K0+LU_OB, n)) in tiles
// of 128 x 32, which = 2 the block-row strip (rows k+LU_NB..min(K0+LU_OB, n), columns
// K0+LU_OB..n) in tiles of 32 x 128: the strips are 32, 64 or 96 wide, so neither
// tile computes padding (64 x 64 tiles did for a quarter of their area; N = 1024, 129
// modes: 41 -> 30 ms).
// 256 threads with 4 x 4 outputs each; bound by FP32 multiply-adds and the tiles'
// loads.
template <int TR, int TC>
__global__ void __launch_bounds__(256) strip_update_kernel(const LuMat* __restrict__ mats, int K0, int k) {
  constexpr bool TALL = TR > TC;
  constexpr int LX = TR / 4;  // threads along the rows: thread x takes rows x + LX a, columns 4 y + c
  const LuMat mat = mats[blockIdx.z];
  const int n = mat.n;
  if (k + LU_NB >= n) return;
  const int bend = min(K0 + LU_OB, n);
  const int r0 = k + LU_NB, r1 = TALL ? n : bend;
  const int c0 = TALL ? k + LU_NB : K0 + LU_OB, c1 = TALL ? bend : n;
  const int i0 = r0 + blockIdx.x * TR, j0 = c0 + blockIdx.y * TC;
  if (i0 >= r1 || j0 >= c1) return;
  cf* M = (cf*)mat.A;
  __shared__ __align__(16) cf As[LU_NB][TR];
  __shared__ __align__(16) cf Bs[LU_NB][TC + 2];
  const int tid = threadIdx.x, tx = tid % LX, ty = tid / LX;
  for (int t = tid; t < LU_NB * TR; t += 256) {
    const int r = t % TR, kk = t / TR;
    As[kk][r] = (i0 + r < r1) ? M[(size_t)(k + kk) * n + i0 + r] : CF(0.f);
  }
  for (int t = tid; t < LU_NB * TC; t += 256) {
    const int kb = t % LU_NB, cj = t / LU_NB;
    Bs[kb][cj] = (j0 + cj < c1) ? M[(size_t)(j0 + cj) * n + k + kb] : CF(0.f);
  }
  __syncthreads();
  cf acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[a][c] = CF(0.f);
#pragma unroll 4
  for (int kk = 0; kk < LU_NB; ++kk) {
    cf av[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) av[a] = As[kk][tx + LX * a];
    const float4 b0 = *(const float4*)&Bs[kk][4 * ty], b1 = *(const float4*)&Bs[kk][4 * ty + 2];
    const cf bv[4] = {CF(b0.x, b0.y), CF(b0.z, b0.w), CF(b1.x, b1.y), CF(b1.z, b1.w)};
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[a][c] = fma(av[a], bv[c], acc[a][c]);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int gj = j0 + 4 * ty + c;
    if (gj >= c1) continue;
    cf* d = M + (size_t)gj * n + i0 + tx;
    cf v[4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (i0 + tx + LX * a < r1) v[a] = d[LX * a];
#pragma unroll
    for (int a = 0; a < 4; ++a)
      if (i0 + tx + LX * a < r1) d[LX * a] = v[a] - acc[a][c];
  }
}

// Tensor-core update of R3: C -= L U with L = A[K0+LU_OB.., K0..K0+LU_OB) and
// U = A[K0..K0+LU_OB, K0+LU_OB..).  Every FP32 operand is split exactly into
// three BF16 pieces (x = hi + mid + lo, 24 bits), and the six piece products
// whose sum carries FP32 precision (hh, hm, mh, hl, mm, lh) are accumulated
// in FP32 tensor memory (-L_im U_im via the MMA's A-negation).  The hi*hi
// products and the five smaller corrections go to separate accumulators (Re
// and Im each, four in all) that are added in registers: sharing one
// accumulator loses about two bits to the tensor core's accumulation, which
// measured 4x the error of a plain FP32 update, while the split form measured
// half of it.  One CTA per 128 x TN output tile of one matrix; 128 threads;
// the operands arrive in LU_OB_CHUNKS chunks of LU_NB k-columns, each in the
// MMA's K-major no-swizzle core-matrix format, through one shared buffer.
#define TCU_M 128
#define TCU_ATILE (TCU_M * LU_NB)  // bf16 elements per piece chunk of an L tile (128 rows x 32 k)

// Column tile TN of the update: 32, 64 or 128 (chosen per block by the tile
// autotuner below).  The update kernel is persistent (one CTA per SM) and
// warp-specialised: a copy thread keeps a ring of NST operand chunks full, an
// MMA thread consumes them into one of NACC accumulator sets in tensor memory
// (4 TN columns each), and four epilogue warps apply a finished tile to C
// while the MMAs of the next tile run.
template <int TN> struct TcuShape {
  static constexpr int BTILE = TN * LU_NB;                        // bf16 elements per piece chunk of a U tile
  static constexpr int STAGE = 6 * (TCU_ATILE + BTILE) * 2;       // one chunk of both operands, six pieces each
  static constexpr int NST = (3 * STAGE <= 220 * 1024) ? 3 : 2;
  static constexpr int SMEM = NST * STAGE;
  static constexpr uint32_t SET_COLS = 4 * TN;
  static constexpr int NACC = (2 * SET_COLS <= 512) ? 2 : 1;
  static constexpr uint32_t TMEM_COLS = NACC * SET_COLS <= 256 ? 256 : 512;
};

__device__ __forceinline__ int tcu_off(int r, int k) {  // 4 core matrices along k
  return ((r >> 3) * (LU_NB / 8) + (k >> 3)) * 64 + (r & 7) * 8 + (k & 7);
}

// Workspace of one matrix: the L block column (rows K0+LU_OB.., LU_OB
// k-columns) and the U block row (LU_OB k-rows, columns K0+LU_OB..) split
// into their BF16 pieces, stored tile by tile in exactly the shared-memory
// image the MMAs read: ceil(n/128) L tiles of [LU_OB_CHUNKS][6 pieces][128 x 32],
// then ceil(n/TN) U tiles of [LU_OB_CHUNKS][6][TN x 32] (room for ceil(n/128)
// tiles of 128 columns, the largest TN).
__host__ __device__ inline size_t tcu_ws_matrix_elems(int n) {
  return (size_t)((n + TCU_M - 1) / TCU_M) * LU_OB_CHUNKS * 6 * (TCU_ATILE + 128 * LU_NB);
}

size_t lu_c64_workspace_bytes(int n, int batch) { return tcu_ws_matrix_elems(n) * (size_t)batch * 2; }

template <int TN>
__global__ void __launch_bounds__(256) tcu_split_kernel(const LuMat* __restrict__ mats, int K0, int nL) {
  using S = TcuShape<TN>;
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n;
  const int start = K0 + LU_OB, rest = n - start;
  if (rest <= 0) return;
  const cf* M = (const cf*)mat.A;
  __nv_bfloat16* W = (__nv_bfloat16*)mat.ws;
  // thread item: one row (of L) or column (of U) and 8 consecutive k, written
  // as one 16-byte core-matrix row per piece
  auto put = [&](__nv_bfloat16* d, int stride, const cf* v) {
    __align__(16) __nv_bfloat16 pc[6][8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      __nv_bfloat16 pr[3], pi[3];
      split3(v[c].x, pr); split3(v[c].y, pi);
#pragma unroll
      for (int q = 0; q < 3; ++q) { pc[q][c] = pr[q]; pc[3 + q][c] = pi[q]; }
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) *(uint4*)(d + (size_t)q * stride) = *(const uint4*)pc[q];
  };
  if ((int)blockIdx.x < nL) {
    if ((int)blockIdx.x * TCU_M >= rest) return;
    const int r0 = start + blockIdx.x * TCU_M;
    __nv_bfloat16* dst = W + (size_t)blockIdx.x * LU_OB_CHUNKS * 6 * TCU_ATILE;
    for (int t = threadIdx.x; t < TCU_M * (LU_OB / 8); t += 256) {
      const int r = t % TCU_M, kb0 = (t / TCU_M) * 8, ch = kb0 / LU_NB, k0 = kb0 % LU_NB;
      cf v[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = (r0 + r < n) ? M[(size_t)(K0 + kb0 + c) * n + r0 + r] : CF(0.f);
      put(dst + (size_t)ch * 6 * TCU_ATILE + tcu_off(r, k0), TCU_ATILE, v);
    }
  } else {
    const int y = blockIdx.x - nL;
    if (y * TN >= rest) return;
    const int c0 = start + y * TN;
    __nv_bfloat16* dst = W + (size_t)((n + TCU_M - 1) / TCU_M) * LU_OB_CHUNKS * 6 * TCU_ATILE +
                         (size_t)y * LU_OB_CHUNKS * 6 * S::BTILE;
    for (int t = threadIdx.x; t < TN * (LU_OB / 8); t += 256) {
      const int kb0 = (t % (LU_OB / 8)) * 8, j = t / (LU_OB / 8), ch = kb0 / LU_NB, k0 = kb0 % LU_NB;
      cf v[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) v[c] = (c0 + j < n) ? M[(size_t)(c0 + j) * n + K0 + kb0 + c] : CF(0.f);
      put(dst + (size_t)ch * 6 * S::BTILE + tcu_off(j, k0), S::BTILE, v);
    }
  }
}

// Persistent update over the tiles of every matrix of the launch: tile t =
// (matrix z, column tile y, row tile x), x fastest, taken by CTA t mod
// gridDim.x; tiles outside a matrix's own trailing block are skipped by all
// three roles alike.  Every wait is bounded: a role that gives up sets the
// CTA's failure flag (and *err), the others stop at their next wait, and
// before the CTA exits the copy thread lets its copies in flight land and the
// MMA thread waits for its MMAs.
template <int TN>
__global__ void __launch_bounds__(192, 1) gemm_update_tc_kernel(const LuMat* __restrict__ mats, int K0, int nLmax,
                                                               int nUmax, int count, int* __restrict__ err) {
  using S = TcuShape<TN>;
  constexpr int NST = S::NST, NACC = S::NACC;
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[NST], empty[NST], tfull[NACC], tempty[NACC], mdone;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  volatile int* fail = &s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int start = K0 + LU_OB;
  const long long per = (long long)nLmax * nUmax, total = per * count;
  auto tile_of = [&](long long t, int& z, int& x, int& y) -> bool {
    z = (int)(t / per);
    const long long r = t - (long long)z * per;
    y = (int)(r / nLmax);
    x = (int)(r - (long long)y * nLmax);
    const int rest = mats[z].n - start;
    return x * TCU_M < rest && y * TN < rest;
  };
  if (warp == 0) tc::tmem_alloc(&tmem_base, S::TMEM_COLS);
  if (tid == 32) {
    s_fail = 0;
#pragma unroll
    for (int b = 0; b < NST; ++b) { tc::mbar_init(&full[b], 1); tc::mbar_init(&empty[b], 1); }
#pragma unroll
    for (int b = 0; b < NACC; ++b) { tc::mbar_init(&tfull[b], 1); tc::mbar_init(&tempty[b], 4); }
    tc::mbar_init(&mdone, 1);
    tc::mbar_fence_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_base;
  int issued = 0;  // copy thread: chunks whose copies were issued
  if (warp == 4) {
    if (lane == 0) {
      int q = 0;
      for (long long t = blockIdx.x; t < total && !*fail; t += gridDim.x) {
        int z, x, y;
        if (!tile_of(t, z, x, y)) continue;
        const int n = mats[z].n;
        const __nv_bfloat16* W = (const __nv_bfloat16*)mats[z].ws;
        const __nv_bfloat16* Lsrc = W + (size_t)x * LU_OB_CHUNKS * 6 * TCU_ATILE;
        const __nv_bfloat16* Usrc = W + (size_t)((n + TCU_M - 1) / TCU_M) * LU_OB_CHUNKS * 6 * TCU_ATILE +
                                    (size_t)y * LU_OB_CHUNKS * 6 * S::BTILE;
        for (int ch = 0; ch < LU_OB_CHUNKS; ++ch, ++q) {
          const int st = q % NST;
          if (q >= NST && !tc::mbar_wait(&empty[st], ((q / NST) - 1) & 1)) { *fail = 1; break; }
          unsigned char* base = smem + (size_t)st * S::STAGE;
          tc::mbar_expect_tx(&full[st], S::STAGE);
          tc::bulk_g2s(base, Lsrc + (size_t)ch * 6 * TCU_ATILE, 6 * TCU_ATILE * 2, &full[st]);
          tc::bulk_g2s(base + 6 * TCU_ATILE * 2, Usrc + (size_t)ch * 6 * S::BTILE, 6 * S::BTILE * 2, &full[st]);
          issued = q + 1;
        }
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {
      const uint32_t id_pos = tc::idesc_bf16_f32(TCU_M, TN, false);
      const uint32_t id_neg = tc::idesc_bf16_f32(TCU_M, TN, true);
      const uint64_t at = (uint64_t)(TCU_ATILE * 2 / 16), bt = (uint64_t)(S::BTILE * 2 / 16);  // 16-byte units
      const int qa_[6] = {0, 0, 1, 0, 1, 2}, qb_[6] = {0, 1, 0, 2, 1, 0};
      int q = 0, k = 0;
      for (long long t = blockIdx.x; t < total && !*fail; t += gridDim.x) {
        int z, x, y;
        if (!tile_of(t, z, x, y)) continue;
        const int set = k % NACC;
        if (k >= NACC && !tc::mbar_wait(&tempty[set], ((k / NACC) - 1) & 1)) { *fail = 1; break; }
        tc::fence_after();
        // accumulator columns of the set: [0,TN) hh Re, [TN,2TN) hh Im, [2TN,3TN) corrections Re, [3TN,4TN) Im
        const uint32_t d0 = tmem + (uint32_t)set * S::SET_COLS;
        for (int ch = 0; ch < LU_OB_CHUNKS; ++ch, ++q) {
          const int st = q % NST;
          if (!tc::mbar_wait(&full[st], (q / NST) & 1)) { *fail = 1; break; }
          tc::fence_after();
          unsigned char* base = smem + (size_t)st * S::STAGE;
          const uint64_t a0 = tc::desc_noswizzle(tc::smem_u32(base), 128, (LU_NB / 8) * 128);
          const uint64_t b0 = tc::desc_noswizzle(tc::smem_u32(base + 6 * TCU_ATILE * 2), 128, (LU_NB / 8) * 128);
#pragma unroll
          for (int ks = 0; ks < LU_NB / 16; ++ks) {
            const uint64_t kof = (uint64_t)(ks * 256 / 16);  // two core matrices along k
#pragma unroll
            for (int u = 0; u < 6; ++u) {
              const uint64_t are = a0 + qa_[u] * at + kof, aim = a0 + (3 + qa_[u]) * at + kof;
              const uint64_t bre = b0 + qb_[u] * bt + kof, bim = b0 + (3 + qb_[u]) * bt + kof;
              const uint32_t dre = d0 + (u == 0 ? 0 : 2 * TN), dim = d0 + (u == 0 ? TN : 3 * TN);
              const uint32_t acc = (ch == 0 && ks == 0 && u <= 1) ? 0u : 1u;  // first write of each accumulator
              tc::mma_bf16(dre, are, bre, id_pos, acc);
              tc::mma_bf16(dre, aim, bim, id_neg, 1u);
              tc::mma_bf16(dim, are, bim, id_pos, acc);
              tc::mma_bf16(dim, aim, bre, id_pos, 1u);
            }
          }
          tc::commit(&empty[st]);  // the stage is free once these MMAs have read it
        }
        if (*fail) break;
        tc::commit(&tfull[set]);   // the tile's accumulators are complete
        ++k;
      }
      tc::commit(&mdone);          // arrives once every MMA issued above has completed
      if (!tc::mbar_wait(&mdone, 0)) *fail = 1;
    }
  } else {
    // epilogue warps: warp w owns tensor-memory lanes (tile rows) 32w .. 32w + 31
    int k = 0;
    for (long long t = blockIdx.x; t < total; t += gridDim.x) {
      int z, x, y;
      if (!tile_of(t, z, x, y)) continue;
      const int set = k % NACC;
      const int n = mats[z].n;
      cf* M = (cf*)mats[z].A;
      const int i = start + x * TCU_M + warp * 32 + lane, j0 = start + y * TN;
      cf cv[32];
#pragma unroll
      for (int c = 0; c < 32; ++c) {  // C of the first 32 columns while the MMAs run
        const int j = j0 + c;
        cv[c] = (i < n && j < n) ? M[(size_t)j * n + i] : CF(0.f);
      }
      if (!tc::mbar_wait(&tfull[set], (k / NACC) & 1)) { *fail = 1; break; }
      tc::fence_after();
      const uint32_t tw = tmem + (uint32_t)set * S::SET_COLS + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
      for (int c0 = 0; c0 < TN; c0 += 32) {
        if (c0 > 0) {
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const int j = j0 + c0 + c;
            cv[c] = (i < n && j < n) ? M[(size_t)j * n + i] : CF(0.f);
          }
        }
        float h[32], e[32];  // Re parts into cv first, then Im: two accumulator pairs live at a time
        tc::tmem_ld32(tw + c0, h);
        tc::tmem_ld32(tw + 2 * TN + c0, e);
#pragma unroll
        for (int c = 0; c < 32; ++c) cv[c].x -= h[c] + e[c];
        tc::tmem_ld32(tw + TN + c0, h);
        tc::tmem_ld32(tw + 3 * TN + c0, e);
#pragma unroll
        for (int c = 0; c < 32; ++c) cv[c].y -= h[c] + e[c];
        if (i < n) {
#pragma unroll
          for (int c = 0; c < 32; ++c) {
            const int j = j0 + c0 + c;
            if (j < n) M[(size_t)j * n + i] = cv[c];
          }
        }
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&tempty[set]);
      ++k;
    }
  }
  __syncthreads();
  if (*fail) {
    if (tid == 0 && err) atomicExch(err, 1);
    if (warp == 4 && lane == 0) {
      // let the copies still in flight land before the CTA exits (bounded):
      // the newest copy of each stage completes the newest phase of its barrier
      for (int st = 0; st < NST; ++st) {
        const int last = issued - 1 - ((issued - 1 - st) % NST + NST) % NST;  // newest chunk issued into st
        if (last >= 0) tc::mbar_wait(&full[st], (last / NST) & 1, 1 << 20);
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, S::TMEM_COLS);
}

// ---------------------------------------------------------------- driver
// R3 of outer block K0 for the matrices 0..active-1 (those with n > K0 + LU_OB);
// rest = nmax - K0 - LU_OB is the largest trailing size.
template <int TN>
static void tc_update_tn(const LuMat* d, int K0, int rest, int active, int* tc_err, cudaStream_t s) {
  const int nL = (rest + TCU_M - 1) / TCU_M, nU = (rest + TN - 1) / TN;
  tcu_split_kernel<TN><<<dim3(nL + nU, active), 256, 0, s>>>(d, K0, nL);
  const long long tiles = (long long)nL * nU * active;
  const int grid = (int)std::min<long long>(tiles, sm_count());
  gemm_update_tc_kernel<TN><<<grid, 192, TcuShape<TN>::SMEM, s>>>(d, K0, nL, nU, active, tc_err);
}

static void tc_update(int tn, const LuMat* d, int K0, int rest, int active, int* tc_err, cudaStream_t s) {
  if (tn == 32) tc_update_tn<32>(d, K0, rest, active, tc_err, s);
  else if (tn == 128) tc_update_tn<128>(d, K0, rest, active, tc_err, s);
  else tc_update_tn<64>(d, K0, rest, active, tc_err, s);
}

static void tc_set_attributes() {
  cudaFuncSetAttribute(gemm_update_tc_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcuShape<32>::SMEM);
  cudaFuncSetAttribute(gemm_update_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcuShape<64>::SMEM);
  cudaFuncSetAttribute(gemm_update_tc_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, TcuShape<128>::SMEM);
}

__global__ void lu_info_zero_kernel(const LuMat* __restrict__ mats, int count) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b < count) mats[b].info[0] = 0;
}

// Tile autotuner.  The column tile TN of the tensor-core update is chosen per
// LU step from the trailing size (rest) and the number of matrices in the
// launch.  For each power-of-two bucket of rest ((64, 128], (128, 256], ...,
// above 8192) and of the matrix count, the split + update pair is timed once
// per process on scratch matrices of the bucket's middle size with TN = 32, 64
// and 128 (CUDA events on the caller's stream, best of three after one
// warm-up); the tile with the least time per matrix is kept, TN = 64 unless
// another is at least 3 % faster.  Scratch is capped near 1 GiB by timing
// fewer matrices of large sizes (their launches still fill the GPU).
namespace {
std::mutex g_tune_mu;
std::map<std::pair<int, int>, int> g_tune;
std::map<std::pair<int, int>, std::array<float, 3>> g_tune_ms;
int rest_bucket(int rest) { int b = 0; while (b < 7 && (128 << b) < rest) ++b; return b; }
int count_bucket(int c) { int b = 0; while (b < 16 && (1 << b) < c) ++b; return b; }
}  // namespace

__global__ void tune_fill_kernel(cf* A, size_t count) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < count; i += (size_t)gridDim.x * blockDim.x) {
    uint32_t h = (uint32_t)(i * 2654435761u) ^ (uint32_t)(i >> 32);
    h ^= h >> 15; h *= 2246822519u; h ^= h >> 13;
    A[i] = CF((float)(h & 0xffff) * (2.f / 65535.f) - 1.f, (float)(h >> 16) * (2.f / 65535.f) - 1.f);
  }
}

static int measure_tile(int R, int count, cudaStream_t s, std::array<float, 3>& ms) {
  const int n = R + LU_OB;
  const size_t elems = (size_t)n * n, wse = tcu_ws_matrix_elems(n);
  const size_t per = elems * sizeof(cf) + wse * 2;
  const int c = (int)std::min<size_t>((size_t)count, std::max<size_t>(1, ((size_t)1 << 30) / per));
  cf* A = nullptr;
  __nv_bfloat16* ws = nullptr;
  LuMat* d = nullptr;
  int* err = nullptr;
  ms = {-1.f, -1.f, -1.f};
  if (cudaMallocAsync((void**)&A, elems * c * sizeof(cf), s) != cudaSuccess ||
      cudaMallocAsync((void**)&ws, wse * c * 2, s) != cudaSuccess ||
      cudaMallocAsync((void**)&d, sizeof(LuMat) * c, s) != cudaSuccess ||
      cudaMallocAsync((void**)&err, sizeof(int), s) != cudaSuccess) {
    cudaGetLastError();
    if (A) cudaFreeAsync(A, s);
    if (ws) cudaFreeAsync(ws, s);
    if (d) cudaFreeAsync(d, s);
    if (err) cudaFreeAsync(err, s);
    return 64;
  }
  std::vector<LuMat> it(c);
  for (int i = 0; i < c; ++i) it[i] = LuMat{A + elems * i, nullptr, nullptr, ws + wse * i, n, 0};
  cudaMemcpyAsync(d, it.data(), sizeof(LuMat) * c, cudaMemcpyHostToDevice, s);
  cudaMemsetAsync(err, 0, sizeof(int), s);
  tune_fill_kernel<<<1024, 256, 0, s>>>(A, elems * c);
  cudaEvent_t e0, e1;
  cudaEventCreate(&e0); cudaEventCreate(&e1);
  const int tns[3] = {32, 64, 128};
  for (int q = 0; q < 3; ++q) {
    tc_update(tns[q], d, 0, R, c, err, s);
    float best = 1e30f;
    for (int rep = 0; rep < 3; ++rep) {
      cudaEventRecord(e0, s);
      tc_update(tns[q], d, 0, R, c, err, s);
      cudaEventRecord(e1, s);
      cudaEventSynchronize(e1);
      float t = 0.f;
      cudaEventElapsedTime(&t, e0, e1);
      best = std::min(best, t);
    }
    ms[q] = best / c;
  }
  int herr = 0;
  cudaMemcpyAsync(&herr, err, sizeof(int), cudaMemcpyDeviceToHost, s);
  cudaStreamSynchronize(s);
  cudaEventDestroy(e0); cudaEventDestroy(e1);
  cudaFreeAsync(A, s); cudaFreeAsync(ws, s); cudaFreeAsync(d, s); cudaFreeAsync(err, s);
  if (cudaGetLastError() != cudaSuccess || herr) return 64;
  int pick = 1;
  for (int q : {0, 2})
    if (ms[q] > 0.f && ms[q] < 0.97f * ms[pick]) pick = q;
  return tns[pick];
}

static void autotune_tiles(int nmax, int count, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  const int cb = count_bucket(count);
  for (int rb = 0; rb <= rest_bucket(nmax - LU_OB); ++rb) {
    if (g_tune.count({rb, cb})) continue;
    std::array<float, 3> ms;
    const int tn = measure_tile(96 << rb, count, s, ms);  // the bucket's middle trailing size
    g_tune[{rb, cb}] = tn;
    g_tune_ms[{rb, cb}] = ms;
  }
}

static int tuned_tile(int rest, int count) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  auto f = g_tune.find({rest_bucket(rest), count_bucket(count)});
  return f == g_tune.end() ? 64 : f->second;
}

int lu_tile_table(int* rest_hi, int* count_hi, int* tile, float* ms, int cap) {
  std::lock_guard<std::mutex> lk(g_tune_mu);
  int k = 0;
  for (const auto& e : g_tune) {
    if (k >= cap) break;
    rest_hi[k] = 128 << e.first.first;
    count_hi[k] = 1 << e.first.second;
    tile[k] = e.second;
    const auto& m = g_tune_ms[e.first];
    for (int q = 0; q < 3; ++q) ms[3 * k + q] = m[q];
    ++k;
  }
  return k;
}

// Complex128 workspace: the matrices (largest first) are factored in groups whose
// luz_matrix_bytes fit the pool; without a pool that holds the largest matrix
// the updates run on the FP64 pipe.
size_t lu_z_pool_bytes(const int* n, int count, size_t most) {
  size_t need = 0, one = 0;
  for (int b = 0; b < count; ++b) {
    const size_t w = luz_matrix_bytes(n[b]);
    need += w;
    one = std::max(one, w);
  }
  return std::max(one, std::min(need, most));
}

// Right-looking blocked LU of every matrix of the table, largest first: at
// step k0 the launches cover the matrices with n > k0 (a prefix of the sorted
// table), each kernel reading its matrix, size and pivots from the table.
// Complex128 with a pool and complex64 work on two levels (LU_NB panels in
// LU_OB blocks, products on the tensor cores); complex128 without a pool
// updates the trailing matrix after every panel on the FP64 pipe.  The choice
// changes rounding, so it is one for all matrices of a call.
template <class T>
static cudaError_t lu_factor_impl(const LuMat* items, int count, cudaStream_t s, LuTiming* tm, int* tc_err, int tile,
                                  bool graph, const LuPool& pool, LuMat* dall) {
  if (count <= 0) return cudaSuccess;
  std::vector<LuMat> it(items, items + count);
  std::stable_sort(it.begin(), it.end(), [](const LuMat& a, const LuMat& b) { return a.n > b.n; });
  constexpr bool c64 = std::is_same<T, cf>::value;
  std::vector<int> groups = {0};  // first matrix of every group
  const bool two_level = c64 || (pool.p && luz_matrix_bytes(it[0].n) <= pool.bytes);
  if (!c64 && two_level) {
    size_t o = 0;
    for (int b = 0; b < count; ++b) {
      const size_t w = luz_matrix_bytes(it[b].n);
      if (o + w > pool.bytes) {
        groups.push_back(b);
        o = 0;
      }
      it[b].ws = (unsigned char*)pool.p + o;
      o += w;
    }
  }
  groups.push_back(count);
  cudaError_t e = cudaSuccess;
  cudaMemcpyAsync(dall, it.data(), sizeof(LuMat) * count, cudaMemcpyHostToDevice, s);
  lu_info_zero_kernel<<<(count + 255) / 256, 256, 0, s>>>(dall, count);
  if constexpr (c64) {
    tc_set_attributes();
    if (tile == 0) autotune_tiles(it[0].n, count, s);
  }
  cudaStream_t ls = s, cs = nullptr;
  // while this thread captures, no other thread of the library frees device
  // memory (a free synchronizes the device, which would end the capture)
  std::unique_lock<std::mutex> capture_lock(lu_capture_mutex(), std::defer_lock);
  if (graph) capture_lock.lock();
  if (graph) {
    if (cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) != cudaSuccess ||
        cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      if (cs) cudaStreamDestroy(cs);
      cs = nullptr;
      graph = false;
      capture_lock.unlock();
    } else {
      ls = cs;
    }
  }
  const bool timed = tm && !graph;
  std::vector<cudaEvent_t> ev;
  int launches = 1, gemm_launches = 0, tn_steps[3] = {0, 0, 0};
  double gemm_flops = 0.0, gemm_bytes = 0.0;
  auto timed_launch = [&](auto&& launch) {
    cudaEvent_t e0 = nullptr, e1 = nullptr;
    if (timed) {
      cudaEventCreate(&e0); cudaEventCreate(&e1);
      cudaEventRecord(e0, ls);
    }
    launch();
    if (timed) {
      cudaEventRecord(e1, ls);
      ev.push_back(e0); ev.push_back(e1);
    }
  };
  for (size_t gi = 0; gi + 1 < groups.size(); ++gi) {
    const LuMat* d = dall + groups[gi];
    const LuMat* g = it.data() + groups[gi];
    int active = groups[gi + 1] - groups[gi];
    const int nmax = g[0].n;
    auto count_update = [&](int k, int K) {  // trailing update of K columns at column k
      for (int b = 0; b < active; ++b) {
        const double rb = (double)(g[b].n - k - K);
        if (rb > 0) {
          gemm_flops += 8.0 * rb * rb * K;
          gemm_bytes += 2.0 * sizeof(T) * rb * rb;   // the trailing matrix read and written once
        }
      }
      ++gemm_launches;
    };
    // one LU_NB panel at column k0: factor, interchange, rows of U right of it
    // (mode 0: all columns; mode 1: within the LU_OB block starting at K0)
    auto panel_step = [&](int k0, int K0, int mode) -> int {
      while (active > 0 && g[active - 1].n <= k0) --active;
      const int nbk = std::min(LU_NB, nmax - k0);
      bool done = false;
      if constexpr (c64) done = launch_panel_reg(d, nmax - k0, k0, active, ls);
      if (!done && !launch_panel_cluster<T>(d, nmax - k0, k0, active, ls))
        panel_kernel<T><<<active, 1024, 0, ls>>>(d, k0);
      ++launches;
      const int hi = mode == 1 ? std::min(K0 + LU_OB, nmax) : nmax;
      if (hi - nbk > 0) {
        swap_kernel<T><<<dim3((hi - nbk + SWAP_COLS - 1) / SWAP_COLS, active), 256, 0, ls>>>(d, k0, K0, mode);
        ++launches;
      }
      const int rest = hi - k0 - nbk;
      if (rest > 0) {
        if constexpr (c64) trsm_c64_kernel<<<dim3((rest + 127) / 128, active), 128, 0, ls>>>(d, k0, K0, mode);
        else if (two_level) luz_panel_rows(d, K0, k0, rest, active, ls);
        else trsm_kernel<<<dim3((rest + 127) / 128, active), 128, 0, ls>>>(d, k0);
        ++launches;
      }
      return rest;
    };
    if (two_level) {
      // LU_NB panels inside LU_OB blocks, one rank-LU_OB tensor-core update per block
      if constexpr (!c64)
        if (nmax > LU_NB) {
          luz_begin(d, nmax, active, ls);
          ++launches;
        }
      for (int K0 = 0; K0 < nmax; K0 += LU_OB) {
        for (int p = 0; p < LU_OB_CHUNKS; ++p) {
          const int k0 = K0 + p * LU_NB;
          if (k0 >= nmax) break;
          const int bcols = panel_step(k0, K0, 1);                    // R1: block columns right of the panel
          if (bcols <= 0) continue;
          const int rows = nmax - k0 - LU_NB;
          if constexpr (c64) {
            strip_update_kernel<128, 32><<<dim3((rows + 127) / 128, (bcols + 31) / 32, active), 256, 0, ls>>>(d, K0, k0);
            ++launches;
          } else {
            launches += luz_panel_update(d, K0, k0, nmax, active, tc_err, ls);
          }
        }
        const int rest = nmax - K0 - LU_OB;                           // columns right of the block
        if (rest <= 0) continue;
        while (active > 0 && g[active - 1].n <= K0 + LU_OB) --active;  // the matrices that have them
        if (active <= 0) continue;
        for (int p = 0; p < LU_OB_CHUNKS; ++p) {                      // the block's interchanges, in order
          swap_kernel<T><<<dim3((rest + SWAP_COLS - 1) / SWAP_COLS, active), 256, 0, ls>>>(d, K0 + p * LU_NB, K0, 2);
          ++launches;
        }
        if constexpr (c64) {
          for (int p = 0; p < LU_OB_CHUNKS; ++p) {                    // rows of U right of the block; R2
            const int k0 = K0 + p * LU_NB;
            trsm_c64_kernel<<<dim3((rest + 127) / 128, active), 128, 0, ls>>>(d, k0, K0, 2);
            ++launches;
            const int brows = LU_OB - (p + 1) * LU_NB;
            if (brows > 0) {
              strip_update_kernel<32, 128><<<dim3((brows + 31) / 32, (rest + 127) / 128, active), 256, 0, ls>>>(
                  d, K0, k0);
              ++launches;
            }
          }
          // R3
          const int tn = tile ? tile : tuned_tile(rest, active);
          timed_launch([&] { tc_update(tn, d, K0, rest, active, tc_err, ls); });
          ++tn_steps[tn == 32 ? 0 : tn == 64 ? 1 : 2];
          launches += 2;
        } else {
          timed_launch([&] { launches += luz_block_update(d, K0, nmax, active, tc_err, ls); });
        }
        count_update(K0, LU_OB);
      }
    } else if constexpr (!c64) {
      for (int k0 = 0; k0 < nmax; k0 += LU_NB) {
        const int rest = panel_step(k0, 0, 0);
        if (rest <= 0) continue;
        const int t = (rest + GT - 1) / GT;
        timed_launch([&] { gemm_update_kernel<<<dim3(t, t, active), 256, 0, ls>>>(d, k0); });
        ++launches;
        count_update(k0, LU_NB);
      }
    }
  }
  if (graph) {
    cudaGraph_t g = nullptr;
    cudaGraphExec_t x = nullptr;
    e = cudaStreamEndCapture(cs, &g);
    capture_lock.unlock();
    if (e == cudaSuccess) e = cudaGraphInstantiate(&x, g, 0);
    if (e == cudaSuccess) e = cudaGraphLaunch(x, s);
    if (x) cudaGraphExecDestroy(x);
    if (g) cudaGraphDestroy(g);
    cudaStreamDestroy(cs);
    if (e != cudaSuccess) {  // nothing of the capture ran: factor with direct launches instead
      cudaGetLastError();
      return lu_factor_impl<T>(items, count, s, tm, tc_err, tile, false, pool, dall);
    }
  }
  if (tm) {
    tm->launches += launches;
    tm->gemm_flops += gemm_flops;
    tm->gemm_bytes += gemm_bytes;
    tm->gemm_launches += gemm_launches;
    tm->graph = graph ? 1 : 0;
    for (int q = 0; q < 3; ++q) tm->tile_steps[q] += tn_steps[q];
    if (!ev.empty()) cudaEventSynchronize(ev.back());
    for (size_t q = 0; q + 1 < ev.size(); q += 2) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[q], ev[q + 1]);
      tm->gemm_ms += ms;
      cudaEventDestroy(ev[q]); cudaEventDestroy(ev[q + 1]);
    }
  }
  return cudaGetLastError();
}

cudaError_t lu_factor_many(const LuMat* items, int count, bool c64, cudaStream_t s, LuTiming* tm, int* tc_err,
                           int tile, bool graph, const LuPool& pool, LuMat* table) {
  return c64 ? lu_factor_impl<cf>(items, count, s, tm, tc_err, tile, graph, pool, table)
             : lu_factor_impl<cd>(items, count, s, tm, tc_err, 0, graph, pool, table);
}

void lu_factor_batched(cd* A, int n, int batch, int* piv, int* info, cudaStream_t s, LuTiming* tm, int* tc_err,
                       const LuPool& pool, LuMat* table) {
  std::vector<LuMat> it(batch);
  for (int b = 0; b < batch; ++b) it[b] = LuMat{A + (size_t)b * n * n, piv + (size_t)b * n, info + b, nullptr, n, 0};
  lu_factor_impl<cd>(it.data(), batch, s, tm, tc_err, 0, false, pool, table);
}

void lu_factor_batched_c64(cf* A, int n, int batch, int* piv, int* info, cudaStream_t s, LuTiming* tm,
                           int* tc_err, void* ws, LuMat* table, int tile) {
  std::vector<LuMat> it(batch);
  for (int b = 0; b < batch; ++b)
    it[b] = LuMat{A + (size_t)b * n * n, piv + (size_t)b * n, info + b,
                  (__nv_bfloat16*)ws + tcu_ws_matrix_elems(n) * b, n, 0};
  lu_factor_impl<cf>(it.data(), batch, s, tm, tc_err, tile, false, LuPool{}, table);
}
