// The contractions of the fields on BF16 tensor cores with FP64 accuracy: the far field
// on a grid, the ring integrals of plane waves, and the fields at points.
//
// Mode m at the polar angles p needs, for the currents X_u (u = 0, 1, 2) of every
// right-hand side, sum_j b_a(p, j) {cos, sin}(p, j) X_u(j) with a = |m + 1|, |m|,
// |m - 1| (ffgrid_mode_kernel forms them on the FP64 pipe). Grouped by a these are
// M + 2 real products: the rows (angle, cos or sin), the columns (u, sign of the
// shifted mode, right-hand side, J or M, Re or Im), the nodes along k. Both operands
// are cut into 8 exact digits of 7 bits (a scale per row and per column), the digit
// products accumulate exactly in tensor memory 256 nodes at a time, the 8 levels
// are joined in 64-bit integers and the chunks added in FP64.
//
// A sum of K terms is off by at most some K 2^-56 max_k |a_k| max_k |b_k| (measured:
// its square root), where an FP64 sum is off by about 2^-53 sum_k |a_k b_k|: less for
// operands of even size, more where the largest entries of row and column do not meet.
// So the nodes' weights, which fall to 1e-9 of the largest toward the axis, go with the
// currents and not with the rows: rows are then at most 1, b_a itself is only known to
// a few 2^-53 of that, and currents near the axis alone keep their digits (weights in
// the rows left errors of 1e-11 of such a field, now 3e-14 and less). Ring samples and cosines are of even
// size. The kernels of a point are not when it is close to the surface: a sum is then
// off by 2^-56 of the largest kernel times the largest current among NF_KC ring points.
// Measured against 80-bit sums from 0.02 of the radius on, currents on the far side
// among them: at most 1.5 times the FP64 pipe's error.
//
// The ring integrals b_a before and the sums over the modes after are contractions
// with cosine tables and go the same way.
//
// FP64 multiply-adds bound the other form (24 per node, mode, angle pair and side in
// the sums over the nodes); here what is left is the samples' sincos, integer work
// and the bytes of the digits. N = 512, M = 64, 8 sides, 180 x 360 directions: ring
// integrals 0.64 -> 0.22 ms, sums over the nodes 2.55 -> 0.48 ms, azimuths 0.47 ->
// 0.15 ms.
#include <algorithm>
#include <cmath>
#include "digits.cuh"
#include "fields_oz.cuh"
#include "fields_plan.cuh"
#include "ozaki.cuh"
#include "smem.cuh"
#include "tc.cuh"

namespace {

#define FFO_STAGE ((FFO_ABLOCK + FFO_BBLOCK) * 2)
#define FFO_NST 4
#define FFO_SET (OZ_S * FFO_NT)             // tensor-memory columns of one accumulator set

// exponent field of the largest |v| seen -> E with |v| / 2^E < 1/2; all zero: 2^E = 2^-1020
__device__ __forceinline__ int scale_exp(unsigned ex) { return (int)max(ex, 1u) - 1021; }
__device__ __forceinline__ unsigned exp_field(double v) { return ((unsigned)__double2hiint(v) >> 20) & 0x7FFu; }
// 2^E; a column with an infinity or NaN gets NaN, which its products then are
__device__ __forceinline__ double scale_of(unsigned ex) {
  return ex == 0x7FFu ? __longlong_as_double(0x7FF8000000000000ll) : ldexp(1.0, scale_exp(ex));
}
// digits of 8 consecutive k of one row: one 16-byte core-matrix row per digit
__device__ __forceinline__ void put_digits(__nv_bfloat16* dst, int stride, const double* v, int E) {
  __align__(16) __nv_bfloat16 pc[OZ_S][8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    int d[OZ_S];
    digits28(fixed_rn(v[c], 56 - E), d);
#pragma unroll
    for (int q = 0; q < OZ_S; ++q) pc[q][c] = __float2bfloat16_rn((float)d[q]);
  }
#pragma unroll
  for (int q = 0; q < OZ_S; ++q) *(uint4*)(dst + (size_t)q * stride) = *(const uint4*)pc[q];
}

// Rows 2 pp + t (t = 0 cos, 1 sin) of index a0 + a for the angles p0 + pp: one CTA per
// (pp - b0, a).  coef: b_{a0 + a} of row (pp - b0) N + j at [index & 1][index / 2][row],
// ldc rows to a column, ncc columns.
__global__ void __launch_bounds__(64) ffo_rows_kernel(int N, int p0, int b0, int a0, int nrt,
                                                      const double* __restrict__ coef, int ncc, size_t ldc,
                                                      const double2* __restrict__ phase,
                                                      __nv_bfloat16* __restrict__ Asl, double* __restrict__ rscale) {
  __shared__ unsigned red[2][2];
  const int pp = b0 + blockIdx.x, a = blockIdx.y, tid = threadIdx.x, nkt = N / OZ_KT;
  const double* b = coef + ((size_t)((a0 + a) & 1) * ncc + ((a0 + a) >> 1)) * ldc + (size_t)blockIdx.x * N;
  const double2* ph = phase + (size_t)(p0 + pp) * N;
  unsigned ex[2] = {0u, 0u};
  for (int j = tid; j < N; j += 64) {
    ex[0] = max(ex[0], exp_field(b[j] * ph[j].x));
    ex[1] = max(ex[1], exp_field(b[j] * ph[j].y));
  }
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    ex[t] = __reduce_max_sync(0xffffffffu, ex[t]);
    if ((tid & 31) == 0) red[t][tid >> 5] = ex[t];
  }
  __syncthreads();
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    ex[t] = max(red[t][0], red[t][1]);
    if (tid == 0) rscale[(size_t)a * nrt * OZ_RT + 2 * pp + t] = scale_of(ex[t]);
  }
  for (int j = 8 * tid; j < N; j += 8 * 64) {  // N is a multiple of 16
    double v[2][8];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const double2 f = ph[j + c];
      v[0][c] = b[j + c] * f.x;
      v[1][c] = b[j + c] * f.y;
    }
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int r = 2 * pp + t, rt = r / OZ_RT, rr = r % OZ_RT;
      put_digits(Asl + (((size_t)a * nrt + rt) * nkt + j / OZ_KT) * FFO_ABLOCK + core_off(rr, j % OZ_KT), FFO_ATILE, v[t],
                 scale_exp(ex[t]));
    }
  }
}

// Columns of mode q and right-hand side w0 + w: X_0 = r' J1 + i J2, X_1 = z' J1,
// X_2 = r' J1 - i J2 (and of M), times the nodes' weights (wt of ffo_phase_kernel), for
// a = |m + 1|, |m|, |m - 1| where that is one of a0 .. a0 + na - 1.  One CTA per (q, w, X).
__global__ void __launch_bounds__(64) ffo_cols_kernel(int N, int M, const double* __restrict__ wt,
                                                      const cd* __restrict__ x, int nrhs, int w0, int nw, int a0,
                                                      int na, int nct, __nv_bfloat16* __restrict__ Bsl,
                                                      double* __restrict__ cscale) {
  __shared__ unsigned red[2];
  const int q = blockIdx.x, w = blockIdx.y, h = blockIdx.z / 3, u = blockIdx.z % 3;
  const int s = q - M + 1 - u, a = abs(s) - a0, nkt = N / OZ_KT, tid = threadIdx.x;
  if (a < 0 || a >= na) return;
  const cd* xv = x + ((size_t)q * nrhs + w0 + w) * 4 * N + 2 * h;
  auto value = [&](int j) {
    const cd v1 = xv[4 * j];
    if (u == 1) return wt[2 * N + j] * v1;
    const cd r1 = wt[N + j] * v1, v2 = wt[j] * mul_i(xv[4 * j + 1]);
    return u == 0 ? r1 + v2 : r1 - v2;
  };
  unsigned ex = 0u;
  for (int j = tid; j < N; j += 64) {
    const cd v = value(j);
    ex = max(ex, max(exp_field(v.x), exp_field(v.y)));
  }
  ex = __reduce_max_sync(0xffffffffu, ex);
  if ((tid & 31) == 0) red[tid >> 5] = ex;
  __syncthreads();
  const unsigned e = max(red[0], red[1]);
  const int col = ((u * 2 + (s < 0)) * nw + w) * 4 + 2 * h, ct = col / FFO_NT, cc = col % FFO_NT;
  if (tid < 2) cscale[((size_t)a * nct) * FFO_NT + col + tid] = scale_of(e);
  __nv_bfloat16* base = Bsl + ((size_t)a * nct + ct) * nkt * FFO_BBLOCK;
  for (int j = 8 * tid; j < N; j += 8 * 64) {
    double re[8], im[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const cd v = value(j + i);
      re[i] = v.x;
      im[i] = v.y;
    }
    __nv_bfloat16* d = base + (size_t)(j / OZ_KT) * FFO_BBLOCK;
    put_digits(d + core_off(cc, j % OZ_KT), FFO_BTILE, re, scale_exp(e));
    put_digits(d + core_off(cc + 1, j % OZ_KT), FFO_BTILE, im, scale_exp(e));
  }
}

// Y[a][column][row] = sum over k of index a's rows and columns, times sc and the
// scales given.  Persistent: CTA b takes the tiles b, b +
// gridDim.x, ... (column tile fastest, then row tile, then a), in chunks of
// OZ_CHUNK k-tiles: warps 0-3 drain a chunk's 8 levels into FP64 sums while the next
// chunk's products run in the other accumulator set; warp 4 copies, warp 5 issues.
// Every wait is bounded; a role that gives up sets the failure flag and *err.
__global__ void __launch_bounds__(192, 1)
    digit_gemm_kernel(const __nv_bfloat16* __restrict__ Asl, const double* __restrict__ rscale,
                    const __nv_bfloat16* __restrict__ Bsl, const double* __restrict__ cscale, double sc, int nkt, int nrt,
                    int nct, long long ntiles, double* __restrict__ Y, int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  uint64_t* full = (uint64_t*)(smem + FFO_NST * FFO_STAGE);
  uint64_t *empty = full + FFO_NST, *tfull = empty + FFO_NST, *tempty = tfull + 2, *mdone = tempty + 2;
  uint32_t* tbase = (uint32_t*)(mdone + 1);
  volatile int* fail = (volatile int*)(tbase + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nch = (nkt + OZ_CHUNK - 1) / OZ_CHUNK;
  if (warp == 0) tc::tmem_alloc(tbase, 512);
  if (tid == 32) {
    *fail = 0;
    for (int b = 0; b < FFO_NST; ++b) { tc::mbar_init(&full[b], 1); tc::mbar_init(&empty[b], 1); }
    for (int b = 0; b < 2; ++b) { tc::mbar_init(&tfull[b], 1); tc::mbar_init(&tempty[b], 4); }
    tc::mbar_init(mdone, 1);
    tc::mbar_fence_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = *tbase;
  int issued = 0;
  if (warp == 4) {
    if (lane == 0) {
      int q = 0;
      for (long long t = blockIdx.x; t < ntiles && !*fail; t += gridDim.x) {
        const long long ar = t / nct, a = ar / nrt;
        const __nv_bfloat16* Ab = Asl + (size_t)ar * nkt * FFO_ABLOCK;
        const __nv_bfloat16* Bb = Bsl + ((size_t)a * nct + t % nct) * nkt * FFO_BBLOCK;
        for (int kt = 0; kt < nkt; ++kt, ++q) {
          const int st = q % FFO_NST;
          if (q >= FFO_NST && !tc::mbar_wait(&empty[st], ((q / FFO_NST) - 1) & 1)) { *fail = 1; break; }
          unsigned char* base = smem + (size_t)st * FFO_STAGE;
          tc::mbar_expect_tx(&full[st], FFO_STAGE);
          tc::bulk_g2s(base, Ab + (size_t)kt * FFO_ABLOCK, FFO_ABLOCK * 2, &full[st]);
          tc::bulk_g2s(base + FFO_ABLOCK * 2, Bb + (size_t)kt * FFO_BBLOCK, FFO_BBLOCK * 2, &full[st]);
          issued = q + 1;
        }
      }
    }
  } else if (warp == 5) {
    if (lane == 0) {
      int q = 0, k = 0;
      for (long long t = blockIdx.x; t < ntiles && !*fail; t += gridDim.x) {
        for (int kt = 0; kt < nkt && !*fail; ++k) {
          const int set = k & 1, kt1 = min(nkt, kt + OZ_CHUNK);
          if (k >= 2 && !tc::mbar_wait(&tempty[set], ((k >> 1) - 1) & 1)) { *fail = 1; break; }
          tc::fence_after();
          const uint32_t acc0 = tmem + (uint32_t)(set * FFO_SET);
          for (bool first = true; kt < kt1; ++kt, ++q, first = false) {
            const int st = q % FFO_NST;
            if (!tc::mbar_wait(&full[st], (q / FFO_NST) & 1)) { *fail = 1; break; }
            tc::fence_after();
            unsigned char* base = smem + (size_t)st * FFO_STAGE;
            const uint64_t a0 = tc::desc_noswizzle(tc::smem_u32(base), 128, 256);
            const uint64_t b0 = tc::desc_noswizzle(tc::smem_u32(base + FFO_ABLOCK * 2), 128, 256);
#pragma unroll
            for (int s = 0; s < OZ_S; ++s)  // digit s times digits 0 .. 7 - s: levels s .. 7; (0, u) opens level u
              tc::mma_bf16(acc0 + (uint32_t)(s * FFO_NT), a0 + (uint64_t)(s * (FFO_ATILE * 2 / 16)), b0,
                           tc::idesc_bf16_f32(OZ_RT, FFO_NT * (OZ_S - s)), (first && s == 0) ? 0u : 1u);
            tc::commit(&empty[st]);
          }
          if (*fail) break;
          tc::commit(&tfull[set]);
        }
      }
      tc::commit(mdone);  // arrives once every MMA issued above has completed
      if (!tc::mbar_wait(mdone, 0)) *fail = 1;
    }
  } else {
    int k = 0;
    bool ok = true;
    for (long long t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      double acc[FFO_NT];
#pragma unroll
      for (int c = 0; c < FFO_NT; ++c) acc[c] = 0.0;
      for (int ch = 0; ch < nch; ++ch, ++k) {
        const int set = k & 1;
        if (!tc::mbar_wait(&tfull[set], (k >> 1) & 1)) { *fail = 1; ok = false; break; }
        tc::fence_after();
        const uint32_t tw = tmem + (uint32_t)(set * FFO_SET) + ((uint32_t)(warp * 32) << 16);
        // levels joined in units of 2^-55 (below 2^63), one FP64 addition per value
#pragma unroll
        for (int h = 0; h < FFO_NT; h += 8) {
          float v[4][8];
          tc::tmem_ld8x4(tw + h, tw + FFO_NT + h, tw + 2 * FFO_NT + h, tw + 3 * FFO_NT + h, v);
          long long hi[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            hi[u] = (long long)(__float2int_rn(v[0][u]) * 128 + __float2int_rn(v[1][u])) * 16384 +
                    (__float2int_rn(v[2][u]) * 128 + __float2int_rn(v[3][u]));
          tc::tmem_ld8x4(tw + 4 * FFO_NT + h, tw + 5 * FFO_NT + h, tw + 6 * FFO_NT + h, tw + 7 * FFO_NT + h, v);
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const long long lo = (long long)(__float2int_rn(v[0][u]) * 128 + __float2int_rn(v[1][u])) * 16384 +
                                 (__float2int_rn(v[2][u]) * 128 + __float2int_rn(v[3][u]));
            acc[h + u] += fixed_to_double(hi[u] * 1048576 + ((lo + 128) >> 8), -55);
          }
        }
        tc::fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive(&tempty[set]);
      }
      if (!ok) break;
      const long long ar = t / nct, a = ar / nrt;
      const int r = warp * 32 + lane;
      const double rs = rscale ? rscale[ar * OZ_RT + r] * sc : sc;
      const double* cs = cscale ? cscale + ((size_t)a * nct + t % nct) * FFO_NT : nullptr;
      double* y = Y + ((size_t)a * nct + t % nct) * FFO_NT * nrt * OZ_RT + (ar % nrt) * OZ_RT + r;
#pragma unroll
      for (int c = 0; c < FFO_NT; ++c) y[(size_t)c * nrt * OZ_RT] = cs ? acc[c] * rs * cs[c] : acc[c] * rs;
    }
  }
  __syncthreads();
  if (*fail) {
    if (tid == 0) atomicExch(err, 1);
    if (warp == 4 && lane == 0) {
      // the copies still in flight land before the CTA exits (bounded)
      for (int st = 0; st < FFO_NST; ++st) {
        const int last = issued - 1 - ((issued - 1 - st) % FFO_NST + FFO_NST) % FFO_NST;  // newest k-tile issued into st
        if (last >= 0) tc::mbar_wait(&full[st], (last / FFO_NST) & 1, 1 << 20);
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// One thread per (angle, mode, right-hand side).
__global__ void __launch_bounds__(128) ffo_vector_kernel(int M, double k0, double omega, cd eps0, int n_polar, int P2,
                                                         int p0, int np, int nrt, int nct, int w0, int nw,
                                                         const double* __restrict__ Y, cd* __restrict__ F) {
  const int pp = blockIdx.x * 128 + threadIdx.x, q = blockIdx.y, m = q - M;
  if (pp >= np) return;
  for (int w = blockIdx.z; w < nw; w += gridDim.z) {
    cd A[6], B[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      const int h = c / 3, u = c % 3, s = m + 1 - u;
      const int col = ((u * 2 + (s < 0)) * nw + w) * 4 + 2 * h;
      const double* y = Y + (((size_t)abs(s) * nct) * FFO_NT + col) * nrt * OZ_RT + 2 * pp;
      const double2 re = *(const double2*)y, im = *(const double2*)(y + (size_t)nrt * OZ_RT);
      A[c] = C(re.x, im.x);
      B[c] = C(re.y, im.y);
    }
    ffgrid_vector(A, B, m, M, k0, omega, eps0, p0 + pp, n_polar, F + (size_t)(w0 + w) * n_polar * (2 * M + 1) * 3);
  }
}

// ---------------------------------------------------------------------------
// Ring integrals b_m(a) = sum_t weight_t {cos, sin}(a cos theta_t) cos(m theta_t) over the
// Q = n / 4 + 1 samples of ring_even_coef, for many arguments a: two real products
// (even and odd m) of the samples' digits with one table of weighted cosines.

// Digits of the table, column c of parity par for m = 2 c + par <= M + 1, and
// cost[t] = cos theta_t.  One CTA per (column, parity); a value per thread, whose cosine
// is a long chain of FP64 operations, then 8 values' digits per thread (M = 64, 65
// samples: 20 -> 6 us against 8 values per thread).
__global__ void __launch_bounds__(128) ring_table_kernel(int M, int n, int nkt, int nct, int E,
                                                         __nv_bfloat16* __restrict__ Bsl, double* __restrict__ cost) {
  __shared__ __align__(16) double v[128];
  const int c = blockIdx.x, par = blockIdx.y, m = 2 * c + par, Q = n / 4 + 1, K = nkt * OZ_KT, tid = threadIdx.x;
  if (c == 0 && par == 0)
    for (int t = tid; t < K; t += 128) cost[t] = t < Q ? cospi(2.0 * t / n) : 0.0;
  if (m > M + 1) return;
  __nv_bfloat16* base = Bsl + ((size_t)par * nct + c / FFO_NT) * nkt * FFO_BBLOCK;
  for (int t0 = 0; t0 < K; t0 += 128) {
    const int t = t0 + tid;
    v[tid] = t < Q ? (t == 0 || t == Q - 1 ? 2.0 : 4.0) / n * cospi(2.0 * (int)((long long)m * t % n) / n) : 0.0;
    __syncthreads();
    const int k = t0 + 8 * tid;
    if (tid < 16 && k < K)
      put_digits(base + (size_t)(k / OZ_KT) * FFO_BBLOCK + core_off(c % FFO_NT, k % OZ_KT), FFO_BTILE, v + 8 * tid, E);
    __syncthreads();
  }
}

// Digits of the samples of 128 rows and 8 consecutive t: row = k N + i has the
// argument scale[k] r_i (scale[k] = k0 d_rho of wave k) or, without scale, (r_i
// sin theta_p) k0 of the polar angle p = p0 + k.
__global__ void __launch_bounds__(128) ring_samples_kernel(const double* __restrict__ r, int N, int nrows,
                                                           const double2* __restrict__ scale, double k0, int p0,
                                                           int n_polar, const double* __restrict__ cost, int nkt, int nrt,
                                                           __nv_bfloat16* __restrict__ Asl) {
  const int row = blockIdx.x * 128 + threadIdx.x, t0 = 8 * blockIdx.y;
  if (row >= nrows) return;
  const int k = row / N, i = row - k * N;
  double arg;
  if (scale) arg = scale[k].x * r[i];
  else {
    double sth, cth;
    sincospi((p0 + k + 0.5) / n_polar, &sth, &cth);
    arg = r[i] * sth * k0;
  }
  double v[2][8];
#pragma unroll
  for (int c = 0; c < 8; ++c) sincos(arg * cost[t0 + c], &v[1][c], &v[0][c]);
  const size_t o = ((size_t)blockIdx.x * nkt + t0 / OZ_KT) * FFO_ABLOCK + core_off(threadIdx.x, t0 % OZ_KT);
#pragma unroll
  for (int par = 0; par < 2; ++par) put_digits(Asl + (size_t)par * nrt * nkt * FFO_ABLOCK + o, FFO_ATILE, v[par], 1);
}

// Phases e^{-i k0 z_j cos theta_p} of the angles 0..P2 - 1, and wt = the weights
// 2 pi w_j r_j, the same times r' and times z'.
__global__ void __launch_bounds__(128) ffo_phase_kernel(FieldGeom g, double k0, int n_polar, double2* __restrict__ phase,
                                                        double* __restrict__ wt) {
  const int p = blockIdx.x, j = blockIdx.y * 128 + threadIdx.x;
  if (j >= g.N) return;
  double s, c;
  sincos(k0 * (g.z[j] * cospi((p + 0.5) / n_polar)), &s, &c);
  phase[(size_t)p * g.N + j] = make_double2(c, -s);
  if (p == 0) {
    const double wr = 6.283185307179586 * g.w[j] * g.r[j];
    wt[j] = wr;
    wt[g.N + j] = wr * g.rp[j];
    wt[2 * g.N + j] = wr * g.zp[j];
  }
}

// ---------------------------------------------------------------------------
// Azimuths of the grid: rows (rhs, polar angle, component, Re or Im) of F_m + F_-m
// (index 0, with cos m phi_s) and i (F_m - F_-m) (index 1, with sin), the modes along k.

// One CTA per (rhs, polar angle) pair: its 6 rows of both indices.
__global__ void __launch_bounds__(128) synth_rows_kernel(int M, const cd* __restrict__ F, int nkt, int nrt,
                                                         __nv_bfloat16* __restrict__ Asl, double* __restrict__ rscale) {
  extern __shared__ __align__(16) double sv[];  // [12][nkt 16], then the rows' largest exponents
  unsigned* ex = (unsigned*)(sv + 12 * nkt * OZ_KT);
  const int K = nkt * OZ_KT, wp = blockIdx.x, tid = threadIdx.x;
  const cd* src = F + (size_t)wp * (2 * M + 1) * 3;
  if (tid < 12) ex[tid] = 0u;
  __syncthreads();
  const int a = tid % 3;
  unsigned mx[4] = {0u, 0u, 0u, 0u};
  for (int m = tid / 3; m < K && tid < 126; m += 42) {
    cd sm = C(0.0), dm = C(0.0);
    if (m <= M) {
      const cd u = src[(M + m) * 3 + a], v = src[(M - m) * 3 + a];
      sm = m ? u + v : u;
      dm = mul_i(u - v);
    }
    const double v[4] = {sm.x, sm.y, dm.x, dm.y};
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sv[((c >> 1) * 6 + 2 * a + (c & 1)) * K + m] = v[c];
      mx[c] = max(mx[c], exp_field(v[c]));
    }
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) atomicMax(&ex[(c >> 1) * 6 + 2 * a + (c & 1)], mx[c]);
  __syncthreads();
  for (int it = tid; it < 12 * (K / 8); it += 128) {
    const int row = it % 12, k = (it / 12) * 8, b = row / 6;
    const long long r = 6ll * wp + row % 6;
    put_digits(Asl + (((size_t)b * nrt + r / OZ_RT) * nkt + k / OZ_KT) * FFO_ABLOCK + core_off((int)(r % OZ_RT), k % OZ_KT),
               FFO_ATILE, sv + row * K + k, scale_exp(ex[row]));
  }
  if (tid < 12) rscale[(size_t)(tid / 6) * nrt * OZ_RT + 6ll * wp + tid % 6] = scale_of(ex[tid]);
}

// cos and sin of m phi_s, column s = 0..n_azim / 2.  One CTA per (column, index), a value
// per thread.
__global__ void __launch_bounds__(128) synth_table_kernel(int M, int n, int nkt, int nct, __nv_bfloat16* __restrict__ Bsl) {
  __shared__ __align__(16) double v[128];
  const int s = blockIdx.x, b = blockIdx.y, K = nkt * OZ_KT, tid = threadIdx.x;
  __nv_bfloat16* base = Bsl + ((size_t)b * nct + s / FFO_NT) * nkt * FFO_BBLOCK;
  for (int m0 = 0; m0 < K; m0 += 128) {
    const int m = m0 + tid;
    const double x = 2.0 * (int)((long long)m * s % n) / n;
    v[tid] = m > M ? 0.0 : b ? sinpi(x) : cospi(x);
    __syncthreads();
    const int k = m0 + 8 * tid;
    if (tid < 16 && k < K)
      put_digits(base + (size_t)(k / OZ_KT) * FFO_BBLOCK + core_off(s % FFO_NT, k % OZ_KT), FFO_BTILE, v + 8 * tid, 1);
    __syncthreads();
  }
}

// Both azimuths s and n - s of a sum, turned into Cartesian components.
__global__ void __launch_bounds__(128) synth_join_kernel(int n_azim, const double* __restrict__ Y, size_t ldy,
                                                         int nct, cd* __restrict__ E) {
  const int s = blockIdx.y * 128 + threadIdx.x, wp = blockIdx.x;
  if (s > n_azim / 2) return;
  cd a[3], b[3];
#pragma unroll
  for (int u = 0; u < 3; ++u) {
    const double2 x = *(const double2*)(Y + (size_t)s * ldy + 6ll * wp + 2 * u);
    const double2 y = *(const double2*)(Y + ((size_t)nct * FFO_NT + s) * ldy + 6ll * wp + 2 * u);
    a[u] = C(x.x, x.y);
    b[u] = C(y.x, y.y);
  }
  for (int mir = 0; mir < 2; ++mir) {
    const int sm = mir ? n_azim - s : s;
    if (mir && (s == 0 || sm == s)) break;
    double sn, cs;
    sincospi(2.0 * sm / n_azim, &sn, &cs);
    const cd v0 = mir ? a[0] - b[0] : a[0] + b[0], v1 = mir ? a[1] - b[1] : a[1] + b[1];
    cd* dst = E + ((size_t)wp * n_azim + sm) * 3;
    dst[0] = cs * v0 - sn * v1;
    dst[1] = sn * v0 + cs * v1;
    dst[2] = mir ? a[2] - b[2] : a[2] + b[2];
  }
}

// ---------------------------------------------------------------------------
// Fields at points: with c1 = G (ik - 1/R), aa = k^2 G + c1/R and bb = -(aa + 2 c1/R)
// curl curl S V = sum T V, T = aa I + bb h h^T (h = R / |R|), curl S V = sum g x V, g = c1 h:
// 18 real rows a point (T_xx, T_yy, T_zz, T_xy, T_xz, T_yz, g; Re, Im), the current
// components as columns (rhs, J or M, component, Re or Im), the ring points along k, cut
// into indices a of NF_KC points each so that few points still fill the device; the
// indices' sums are added in FP64. The kernels of a (point, ring point) pair remain
// FP64 work (about 100 operations) and bound the call, their products with the
// currents (104 operations per right-hand side in nearfield_kernel) do not: N = 320,
// M = 32, 2 sides, 100 points 2.74 -> 1.61 ms, of which kernels 0.87 and products 0.34.
#define NF_LD (NF_KC + 2)

// One CTA per (index a0 + blockIdx.x, point p0 + blockIdx.y): the rows of NF_KC ring
// points through shared memory.
__global__ void __launch_bounds__(128) nf_rows_kernel(long long total, const double4* __restrict__ pts,
                                                      const double* __restrict__ X, int a0, int p0, cd k, int nrt,
                                                      __nv_bfloat16* __restrict__ Asl, double* __restrict__ rscale) {
  extern __shared__ __align__(16) double sv[];  // [NF_ROWS][NF_LD], then the rows' largest exponents
  unsigned* ex = (unsigned*)(sv + NF_ROWS * NF_LD);
  const int a = blockIdx.x, pp = blockIdx.y, tid = threadIdx.x;
  const double x0 = X[3 * (p0 + pp)], x1 = X[3 * (p0 + pp) + 1], x2 = X[3 * (p0 + pp) + 2];
  if (tid < NF_ROWS) ex[tid] = 0u;
  __syncthreads();
  unsigned mx[NF_ROWS];
#pragma unroll
  for (int t = 0; t < NF_ROWS; ++t) mx[t] = 0u;
  const bool lossless = k.y == 0.0;
  const cd k2 = k * k;
#pragma unroll 1
  for (int u = 0; u < NF_KC / 128; ++u) {
    const int col = tid + 128 * u;
    const long long it = (long long)(a0 + a) * NF_KC + col;
    cd T[9];
    if (it < total) {
      const double4 y = pts[it];
      const double R0 = x0 - y.x, R1 = x1 - y.y, R2 = x2 - y.z;
      const double R = sqrt(R0 * R0 + R1 * R1 + R2 * R2), iR = 1.0 / R;
      const double h0 = R0 * iR, h1 = R1 * iR, h2 = R2 * iR;
      double sn, cs;
      sincos(k.x * R, &sn, &cs);
      double am = y.w * iR;  // 1 / 4 pi with the sums
      if (!lossless) am *= exp(-(k.y * R));
      const cd G = C(am * cs, am * sn);
      const cd c1 = lossless ? C(-(G.x * iR + G.y * k.x), G.x * k.x - G.y * iR) : G * C(-k.y - iR, k.x);
      const cd w1 = iR * c1;
      const cd aa = lossless ? fma(k2.x, G, w1) : fma(k2, G, w1);
      const cd nb = fma(2.0, w1, aa);
      const cd n0 = h0 * nb, n1 = h1 * nb, n2 = h2 * nb;
      T[0] = fma(-h0, n0, aa); T[1] = fma(-h1, n1, aa); T[2] = fma(-h2, n2, aa);
      T[3] = -h0 * n1; T[4] = -h0 * n2; T[5] = -h1 * n2;
      T[6] = h0 * c1; T[7] = h1 * c1; T[8] = h2 * c1;
    } else {
#pragma unroll
      for (int t = 0; t < 9; ++t) T[t] = C(0.0);
    }
#pragma unroll
    for (int t = 0; t < 9; ++t) {
      sv[2 * t * NF_LD + col] = T[t].x;
      sv[(2 * t + 1) * NF_LD + col] = T[t].y;
      mx[2 * t] = max(mx[2 * t], exp_field(T[t].x));
      mx[2 * t + 1] = max(mx[2 * t + 1], exp_field(T[t].y));
    }
  }
#pragma unroll
  for (int t = 0; t < NF_ROWS; ++t) {
    const unsigned e = __reduce_max_sync(0xffffffffu, mx[t]);
    if ((tid & 31) == 0) atomicMax(&ex[t], e);
  }
  __syncthreads();
  const int r0 = NF_ROWS * pp;
  for (int i = tid; i < NF_ROWS * (NF_KC / 8); i += 128) {  // rows fastest: neighbouring core-matrix rows
    const int t = i % NF_ROWS, c = (i / NF_ROWS) * 8, r = r0 + t;
    put_digits(Asl + (((size_t)a * nrt + r / OZ_RT) * (NF_KC / OZ_KT) + c / OZ_KT) * FFO_ABLOCK +
                   core_off(r % OZ_RT, c % OZ_KT),
               FFO_ATILE, sv + t * NF_LD + c, scale_exp(ex[t]));
  }
  if (tid < NF_ROWS) rscale[(size_t)a * nrt * OZ_RT + r0 + tid] = scale_of(ex[tid]);
}

// Columns of one right-hand side's currents cur[w0 + w][it][J 3, M 3].  One CTA per
// (index a0 + blockIdx.x, w).
__global__ void __launch_bounds__(64) nf_cols_kernel(long long total, const cd* __restrict__ cur, int a0, int w0, int nct,
                                                     __nv_bfloat16* __restrict__ Bsl, double* __restrict__ cscale) {
  __shared__ unsigned red[12][2];
  const int a = blockIdx.x, w = blockIdx.y, tid = threadIdx.x;
  const long long it0 = (long long)(a0 + a) * NF_KC + 8 * tid;  // total is a multiple of 16
  const bool in = it0 < total;
  const cd* src = cur + ((size_t)(w0 + w) * total + it0) * 6;
  unsigned mx[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) mx[c] = 0u;
  if (in)
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int c = 0; c < 6; ++c) {
        const cd v = src[6 * i + c];
        mx[2 * c] = max(mx[2 * c], exp_field(v.x));
        mx[2 * c + 1] = max(mx[2 * c + 1], exp_field(v.y));
      }
#pragma unroll
  for (int c = 0; c < 12; ++c) {
    mx[c] = __reduce_max_sync(0xffffffffu, mx[c]);
    if ((tid & 31) == 0) red[c][tid >> 5] = mx[c];
  }
  __syncthreads();
#pragma unroll 1
  for (int c = 0; c < 12; ++c) {
    const unsigned e = max(red[c][0], red[c][1]);
    const int col = 12 * w + c, cc = col % FFO_NT;
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = in ? ((const double*)src)[12 * i + c] : 0.0;
    put_digits(Bsl + (((size_t)a * nct + col / FFO_NT) * (NF_KC / OZ_KT) + 8 * tid / OZ_KT) * FFO_BBLOCK +
                   core_off(cc, 8 * tid % OZ_KT),
               FFO_BTILE, v, scale_exp(e));
    if (tid == 0) cscale[(size_t)a * nct * FFO_NT + col] = scale_of(e);
  }
}

// Ysum[column][row] = the sum of the indices' Y (add: to what a pass before left there).
__global__ void __launch_bounds__(128) nf_sum_kernel(int na, long long count, bool add, const double* __restrict__ Y,
                                                     double* __restrict__ Ysum) {
  const long long e = (long long)blockIdx.x * 128 + threadIdx.x;
  if (e >= count) return;
  double acc = add ? Ysum[e] : 0.0;
#pragma unroll 8
  for (int a = 0; a < na; ++a) acc += Y[(size_t)a * count + e];
  Ysum[e] = acc;
}

// out[w][p][6]: E = cJ curl curl S J + cM curl S M, H = dM curl curl S M + dJ curl S J.
__global__ void __launch_bounds__(128) nf_join_kernel(int np, int p0, int nt, int nw, size_t ldy,
                                                      const double* __restrict__ Ysum, cd cJ, cd cM, cd dM, cd dJ,
                                                      cd* __restrict__ out) {
  const long long t = (long long)blockIdx.x * 128 + threadIdx.x;
  if (t >= (long long)nw * np * 6) return;
  const int c = (int)(t % 6), pp = (int)(t / 6 % np), w = (int)(t / 6 / np), i = c % 3, j = (i + 1) % 3, l = (i + 2) % 3;
  const int sym[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
  // row type r (complex) times component v of current h
  auto prod = [&](int r, int h, int v) {
    const double* y = Ysum + (size_t)(12 * w + 6 * h + 2 * v) * ldy + NF_ROWS * pp + 2 * r;
    return C(y[0] - y[ldy + 1], y[ldy] + y[1]);
  };
  const int hc = c < 3 ? 0 : 1, hu = 1 - hc;  // E: curl curl of J, curl of M; H: the other way round
  const cd cc = (prod(sym[i][i], hc, i) + prod(sym[i][j], hc, j)) + prod(sym[i][l], hc, l);
  const cd cu = prod(6 + j, hu, l) - prod(6 + l, hu, j);
  const double inv4pi = 1.0 / (4.0 * 3.141592653589793);
  out[((size_t)w * nt + p0 + pp) * 6 + c] = inv4pi * (c < 3 ? cJ * cc + cM * cu : dM * cc + dJ * cu);
}

// The SMs of the device. Kernel limits and queries come before a call's first launch:
// an attribute call between launches clears the error of a launch that failed.
int digit_ready() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  smem_optin(digit_gemm_kernel);
  smem_optin(synth_rows_kernel);
  smem_optin(nf_rows_kernel);
  return sms;
}

void digit_gemm(int sms, const __nv_bfloat16* Asl, const double* rscale, const __nv_bfloat16* Bsl, const double* cscale,
                double sc, int nkt, int nrt, int nct, int na, double* Y, int* err, cudaStream_t s) {
  const long long ntiles = (long long)na * nrt * nct;
  digit_gemm_kernel<<<(int)std::min<long long>(ntiles, sms), 192, FFO_NST * FFO_STAGE + 256, s>>>(
      Asl, rscale, Bsl, cscale, sc, nkt, nrt, nct, ntiles, Y, err);
}

void ring_table(const RingPlan& f, int M, int n, __nv_bfloat16* Bsl, double* cost, cudaStream_t s) {
  ring_table_kernel<<<dim3(f.nct * FFO_NT, 2), 128, 0, s>>>(M, n, f.nkt, f.nct, f.E, Bsl, cost);
}
void ring_integrals(int sms, const RingPlan& f, const FieldGeom& g, int count, const double2* scale, double k0, int p0, int n_polar,
                    __nv_bfloat16* Asl, const __nv_bfloat16* Bsl, const double* cost, double* Y, int* err, cudaStream_t s) {
  const int nrows = count * g.N, nrt = (int)tiles(nrows, OZ_RT);
  ring_samples_kernel<<<dim3(nrt, 2 * f.nkt), 128, 0, s>>>(g.r, g.N, nrows, scale, k0, p0, n_polar, cost, f.nkt, nrt, Asl);
  digit_gemm(sms, Asl, nullptr, Bsl, nullptr, ldexp(1.0, 1 + f.E), f.nkt, nrt, f.nct, 2, Y, err, s);
}

// Modal data of plane waves from the ring integrals (the formulas of rhs_kernel): rows
// w N + i of coef, one thread per (node, wave) and a run of qc modes m >= 0.  The table
// without the traces' factors has u_0(-m) = s conj u_2(m), u_1(-m) = -s conj u_1(m),
// u_2(-m) = s conj u_0(m), s = (-1)^(m+1) (real polarisations), so the sums of m give
// those of -m: 63 FP64 operations for both modes, both traces of E and of H, where the
// modes by themselves take 78 (N = 512, M = 64, 96 waves: 0.59 -> 0.55 ms).
template <bool ALIGNED>
__global__ void __launch_bounds__(128) rhs_rows_kernel(FieldGeom g, int M, const double2* __restrict__ wave,
                                                       const cd* __restrict__ tab, cd fE, cd fH,
                                                       const double* __restrict__ coef, int ncc, size_t ldc, int w0,
                                                       int nrhs, int qc, cd* __restrict__ rhs) {
  const int w = blockIdx.x, i = blockIdx.y * 128 + threadIdx.x, m0 = blockIdx.z * qc, m1 = min(m0 + qc, M + 1);
  if (i >= g.N) return;
  double s, c;
  sincos(wave[w].y * g.z[i], &s, &c);
  const cd F[2] = {fE * C(c, s), fH * C(c, s)};
  const double rp = g.rp[i], zp = g.zp[i];
  const double* row = coef + (size_t)w * g.N + i;
  auto b = [&](int m) {
    const int a = abs(m);
    return row[((size_t)(a & 1) * ncc + (a >> 1)) * ldc];
  };
  auto put = [&](cd* o, cd o0, cd o1) {
    if (ALIGNED) {
      ((double2*)o)[0] = make_double2(o0.x, o0.y);
      ((double2*)o)[1] = make_double2(o1.x, o1.y);
    } else {
      o[0] = o0;
      o[1] = o1;
    }
  };
  const size_t ld = (size_t)nrhs * 4 * g.N;  // a mode
  cd* o = rhs + (size_t)(w0 + w) * (4 * g.N) + 4 * i;
  double bl = b(m0 - 1), b0 = b(m0);
  for (int m = m0; m < m1; ++m) {
    const double bh = b(m + 1);
    const double rl = rp * bl, rh = rp * bh, z0 = zp * b0;
    const cd* u = tab + ((size_t)w * (2 * M + 1) + M + m) * 6;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const cd u0 = u[3 * h], u1 = u[3 * h + 1], u2 = u[3 * h + 2];
      const cd d = C(fma(bl, u0.x, -(bh * u2.x)), fma(bl, u0.y, -(bh * u2.y)));
      const cd A = C(fma(rl, u0.x, rh * u2.x), fma(rl, u0.y, rh * u2.y)), G = z0 * u1;
      put(o + (size_t)(M + m) * ld + 2 * h, mul_i(d * F[h]), -((A + G) * F[h]));
      if (m > 0) {
        const cd p = conj(d) * F[h], q = conj(A - G) * F[h];  // times -s and s
        put(o + (size_t)(M - m) * ld + 2 * h, m & 1 ? C(p.y, -p.x) : mul_i(p), m & 1 ? -q : q);
      }
    }
    bl = b0;
    b0 = bh;
  }
}

}  // namespace

void launch_ffgrid_products(const FieldGeom& g, int M, double k0, double omega, cd eps0, const cd* x, int nrhs,
                            int n_polar, int n_azim, int n_alpha, const FfoPlan& f, void* work, cd* F, cd* E, int* err,
                            cudaStream_t s) {
  const int sms = digit_ready();
  char* p = (char*)work;
  auto* phase = (double2*)(p + f.phase);
  auto* wt = (double*)(phase + (size_t)f.P2 * g.N);
  auto* Asl = (__nv_bfloat16*)(p + f.a);
  auto* rscale = (double*)(p + f.r);
  auto* Bsl = (__nv_bfloat16*)(p + f.b);
  auto* cscale = (double*)(p + f.c);
  auto* Y = (double*)(p + f.y);
  auto* Tsl = (__nv_bfloat16*)(p + f.table);
  auto* cost = (double*)(p + f.cost);
  auto coef = [&](int b0) { return (double*)(p + f.coef + b0 / f.nps * f.coef_block); };  // of the block at angle b0
  ffo_phase_kernel<<<dim3(f.P2, (g.N + 127) / 128), 128, 0, s>>>(g, k0, n_polar, phase, wt);
  ring_table(f.ring, M, n_alpha, Tsl, cost, s);
  for (int p0 = 0; p0 < f.P2; p0 += f.np) {
    const int np = std::min(f.np, f.P2 - p0), nrt = (int)tiles((size_t)2 * np, OZ_RT);
    for (int b0 = 0; b0 < np; b0 += f.nps)
      ring_integrals(sms, f.ring, g, std::min(f.nps, np - b0), nullptr, k0, p0 + b0, n_polar, Asl, Tsl, cost, coef(b0),
                     err, s);
    for (int w0 = 0; w0 < nrhs; w0 += f.nw) {
      const int nw = std::min(f.nw, nrhs - w0), nct = (int)tiles((size_t)24 * nw, FFO_NT);
      for (int a0 = 0; a0 < f.na; a0 += f.nap) {
        const int na = std::min(f.nap, f.na - a0);
        if (w0 == 0 || f.nap < f.na)  // else the rows' digits are still there
          for (int b0 = 0; b0 < np; b0 += f.nps) {
            const int nb = std::min(f.nps, np - b0);
            ffo_rows_kernel<<<dim3(nb, na), 64, 0, s>>>(g.N, p0, b0, a0, nrt, coef(b0), f.ring.nct * FFO_NT,
                                                        tiles((size_t)nb * g.N, OZ_RT) * OZ_RT, phase, Asl, rscale);
          }
        ffo_cols_kernel<<<dim3(2 * M + 1, nw, 6), 64, 0, s>>>(g.N, M, wt, x, nrhs, w0, nw, a0, na, nct, Bsl, cscale);
        digit_gemm(sms, Asl, rscale, Bsl, cscale, 1.0, f.nkt, nrt, nct, na, Y + (size_t)a0 * nct * FFO_NT * nrt * OZ_RT,
                   err, s);
      }
      ffo_vector_kernel<<<dim3((np + 127) / 128, 2 * M + 1, std::min(nw, 64)), 128, 0, s>>>(
          M, k0, omega, eps0, n_polar, f.P2, p0, np, nrt, nct, w0, nw, Y, F);
    }
  }
  synth_table_kernel<<<dim3(n_azim / 2 + 1, 2), 128, 0, s>>>(M, n_azim, f.snkt, f.snct, Bsl);
  const long long pairs = (long long)nrhs * n_polar;
  for (long long q0 = 0; q0 < pairs; q0 += f.swp) {
    const int nq = (int)std::min<long long>(f.swp, pairs - q0), nrt = (int)tiles((size_t)6 * nq, OZ_RT);
    synth_rows_kernel<<<nq, 128, 12 * (f.snkt * OZ_KT * 8 + 4), s>>>(M, F + (size_t)q0 * (2 * M + 1) * 3, f.snkt, nrt,
                                                                     Asl, rscale);
    digit_gemm(sms, Asl, rscale, Bsl, nullptr, 2.0, f.snkt, nrt, f.snct, 2, Y, err, s);
    synth_join_kernel<<<dim3(nq, (n_azim / 2 + 128) / 128), 128, 0, s>>>(n_azim, Y, (size_t)nrt * OZ_RT, f.snct,
                                                                         E + (size_t)q0 * n_azim * 3);
  }
}

void launch_rhs_products(const FieldGeom& g, int M, const double2* wave, const cd* tab, cd fE, cd fH, int w0, int count,
                         int nrhs, int n_theta, const RhsPlan& plan, void* work, cd* rhs, int* err, cudaStream_t s) {
  const RingPlan& f = plan.ring;
  const int sms = digit_ready();
  const int nw = plan.waves;
  auto* Asl = (__nv_bfloat16*)((char*)work + plan.a);
  auto* Tsl = (__nv_bfloat16*)((char*)work + plan.table);
  auto* cost = (double*)((char*)work + plan.cost);
  auto* coef = (double*)((char*)work + plan.coef);
  ring_table(f, M, n_theta, Tsl, cost, s);
  for (int v0 = 0; v0 < count; v0 += nw) {
    const int c = std::min(nw, count - v0), nb = (g.N + 127) / 128;
    ring_integrals(sms, f, g, c, wave + v0, 0.0, 0, 0, Asl, Tsl, cost, coef, err, s);
    // runs of modes: some 40000 threads in all, at least two pairs of modes each
    const int runs = std::max(1, std::min((M + 2) / 2, 320 / (nb * c) + 1)), qc = (M + runs) / runs;
    const dim3 grid(c, nb, (M + qc) / qc);
    const size_t ldc = tiles((size_t)c * g.N, OZ_RT) * OZ_RT;
    const cd* t = tab + (size_t)v0 * (2 * M + 1) * 6;
    if (((size_t)rhs & 15) == 0)
      rhs_rows_kernel<true><<<grid, 128, 0, s>>>(g, M, wave + v0, t, fE, fH, coef, f.nct * FFO_NT, ldc, w0 + v0, nrhs, qc, rhs);
    else
      rhs_rows_kernel<false><<<grid, 128, 0, s>>>(g, M, wave + v0, t, fE, fH, coef, f.nct * FFO_NT, ldc, w0 + v0, nrhs, qc, rhs);
  }
}

void launch_nearfield_products(long long total, const double4* pts, const cd* cur, const double* X, int nt, int nrhs,
                               cd k, cd cJ, cd cM, cd dM, cd dJ, const NfPlan& f, void* work, cd* out, int* err,
                               cudaStream_t s) {
  const int sms = digit_ready();
  char* p = (char*)work;
  auto* Asl = (__nv_bfloat16*)(p + f.a);
  auto* rscale = (double*)(p + f.r);
  auto* Bsl = (__nv_bfloat16*)(p + f.b);
  auto* cscale = (double*)(p + f.c);
  auto* Y = (double*)(p + f.y);
  auto* Ysum = (double*)(p + f.sum);
  const int vs = f.groups * f.nw, qs = f.passes * f.np;
  for (int v0 = 0; v0 < nrhs; v0 += vs)
    for (int q0 = 0; q0 < nt; q0 += qs) {
      const int v1 = std::min(nrhs, v0 + vs), q1 = std::min(nt, q0 + qs);
      const bool kept = v1 - v0 <= f.nw;  // one product's columns: their digits serve every point
      auto sums = [&](int p0, int w0) { return Ysum + ((size_t)((p0 - q0) / f.np) * f.groups + (w0 - v0) / f.nw) * f.sum_group; };
      for (int a0 = 0; a0 < f.na; a0 += f.nap) {
        const int na = std::min(f.nap, f.na - a0);
        for (int p0 = q0; p0 < q1; p0 += f.np) {
          const int np = std::min(f.np, q1 - p0), nrt = (int)tiles((size_t)NF_ROWS * np, OZ_RT);
          nf_rows_kernel<<<dim3(na, np), 128, NF_ROWS * (NF_LD * 8 + 4), s>>>(total, pts, X, a0, p0, k, nrt, Asl, rscale);
          for (int w0 = v0; w0 < v1; w0 += f.nw) {
            const int nw = std::min(f.nw, v1 - w0), nct = (int)tiles((size_t)12 * nw, FFO_NT);
            if (!kept || p0 == q0) nf_cols_kernel<<<dim3(na, nw), 64, 0, s>>>(total, cur, a0, w0, nct, Bsl, cscale);
            digit_gemm(sms, Asl, rscale, Bsl, cscale, 1.0, NF_KC / OZ_KT, nrt, nct, na, Y, err, s);
            const long long count = (long long)nct * FFO_NT * nrt * OZ_RT;
            nf_sum_kernel<<<(unsigned)((count + 127) / 128), 128, 0, s>>>(na, count, a0 > 0, Y, sums(p0, w0));
          }
        }
      }
      for (int p0 = q0; p0 < q1; p0 += f.np)
        for (int w0 = v0; w0 < v1; w0 += f.nw) {
          const int np = std::min(f.np, q1 - p0), nw = std::min(f.nw, v1 - w0);
          const long long items = (long long)nw * np * 6;
          nf_join_kernel<<<(unsigned)((items + 127) / 128), 128, 0, s>>>(
              np, p0, nt, nw, tiles((size_t)NF_ROWS * np, OZ_RT) * OZ_RT, sums(p0, w0), cJ, cM, dM, dJ,
              out + (size_t)w0 * nt * 6);
        }
    }
}
