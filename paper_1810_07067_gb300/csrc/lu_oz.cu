// FP64-accurate products of the complex128 LU on BF16 tensor cores.
//
// C -= L U (C m x c, inner dimension K = 32 or 128) by exact digit slicing, as in
// ozaki.cu, with the inner dimension graded first: with d_k the power of two
// at the largest entry of row k of U, every row of L D is scaled by its largest
// entry l_ik d_k and every column of D^{-1} U by its largest u_kj / d_k.  Matrices
// whose rows differ by many orders (rows near the axis carry m^2 / r^2) keep
// their small rows this way: the error of an entry is a few 2^-56 of
// max_k |l_ik| d_k max_k |u_kj| / d_k per term, where scaling L and U alone would
// leave that of the product of their unrelated maxima.  That is FP64 accuracy as
// partial pivoting has it, relative to the largest entry of the column of A, wherever
// max_k |l_ik| d_k and max_k |u_kj| / d_k meet near one k.  They need not: rows of U that
// reach into unlike columns have unlike d_k, and a product of small terms then gets the
// error of a large one that is not there (sparse or weakly coupled matrices, columns or
// blocks scaled by 1e8: residuals of 1e-4 of the column).  So a tile whose row and
// column bounds multiply to more than 2^Z_SAFE times a column's largest entry of A is formed
// on the FP64 pipe instead, by the warps that would have drained it.  Gaussian matrices of
// order 64 to 3000 stay at 2^6 and below, those of bodies (sphere, cylinder, cone, torus,
// random, droplet; contrast up to 100) at 2^6 and mostly below 1.  Eight balanced 7-bit
// digits a value, |v| / scale < 1 (the first digit up to 128: the dropped levels
// s + t > 7 are the largest error, and a tighter scale divides them by 4); the
// products of levels s + t <= 7 are exact FP32 integers (at most K 2 (l + 3) 64^2
// < 2^24); a level's sums are joined in 64-bit integers in units of 2^-54 of the
// scales, rounded once to FP64 on the integer pipe, and subtracted from C in
// FP64.
//
// One entry costs 144 digit products per k on the tensor cores and about 60
// integer operations and one FP64 addition per K, where the FP64 pipe (two
// multiply-adds per clock and SM on this part) spends 2 K clocks of an SM on it.
// LU of 9 matrices of order 1250: 69.3 -> 13.2 ms; the cylinder's 65 matrices of order
// 1280: updates 298 -> 12 ms (17 ms with an MMA per pair of digits, which is bound by
// reading the tiles of L again and again: the digits of U lie behind one another, so
// one MMA takes a digit of L times up to four of U into as many levels).  Residuals of
// random factors 1.4e-15 (1.9e-15 on the FP64 pipe), of diagonally dominant ones 1.7e-16
// (1.9e-16).
//
// The block row U12 = L11^{-1} A12 of a 128-column block: four FP64 triangular
// solves of 32 rows, the rows below updated by products with the tile roles
// swapped (tile rows = matrix columns), since the block has at most 96 of them.
// (One product with an explicit L11^{-1} was as fast and left twice the residual
// on random matrices.)
#include <algorithm>
#include <cuda_bf16.h>
#include "cplx.cuh"
#include "digits.cuh"
#include "lu_oz.cuh"
#include "smem.cuh"
#include "tc.cuh"

#define ZR 128                                  // rows of an output tile
#define ZC 32                                   // columns of an output tile
#define ZK 16                                   // inner dimension of a k-tile
#define ZKT (ZB / ZK)                           // k-tiles of a full block
#define ZA_TILE (ZR * ZK)                       // bf16 elements of one digit of one part
#define ZA_BLOCK (2 * OZ_S * ZA_TILE)           // [Re, Im][digit] of a k-tile
#define ZB_TILE (ZC * ZK)
#define ZB_BLOCK (4 * OZ_S * ZB_TILE)           // [digit][Re, Im], then [digit][-Im, Re]
#define Z_STAGE ((ZA_BLOCK + ZB_BLOCK) * 2)     // bytes of a k-tile of both operands
#define Z_NST 2
#define Z_DRAIN 16                              // drain warps of the product
#define Z_THREADS (32 * (Z_DRAIN + 2))
#define Z_NAN (1 << 28)                         // exponent that marks a row or column with Inf or NaN
#define Z_NONE (-(1 << 24))                     // of a row or column of zeros
#define Z_SAFE 8                                // largest exponent of a tile's bound over its columns' entries of A

// Workspace of a matrix: digits of up to ceil(n/128) row tiles and ceil(n/32)
// column tiles, their scale exponents, the high words of the largest
// magnitude in each row of U12, the exponents of the largest entry of each column of A,
// and the largest of a tile's scale exponents (those of columns of U less the column's).
struct ZWork {
  __nv_bfloat16 *Ad, *Bd;
  int *rowE, *colE;
  unsigned* dmax;  // [ZB]
  int *colA, *rowT, *colT;
};
__host__ __device__ inline size_t z_up(size_t b) { return (b + 255) & ~(size_t)255; }
__host__ __device__ inline int z_tiles(int n, int t) { return (n + t - 1) / t; }
__host__ __device__ inline size_t z_bytes(int n, ZWork* w, unsigned char* base) {
  const size_t nr = z_tiles(n, ZR), nc = z_tiles(n, ZC);
  size_t o = 0;
  auto take = [&](size_t b) { const size_t p = o; o += z_up(b); return p; };
  const size_t oa = take(nr * ZKT * ZA_BLOCK * 2), ob = take(nc * ZKT * ZB_BLOCK * 2);
  const size_t orr = take(nr * ZR * 4), oc = take(nc * ZC * 4), od = take(ZB * 4);
  const size_t oca = take((size_t)n * 4), ort = take(nr * 4), oct = take(nc * 4);
  if (w) {
    w->Ad = (__nv_bfloat16*)(base + oa); w->Bd = (__nv_bfloat16*)(base + ob);
    w->rowE = (int*)(base + orr); w->colE = (int*)(base + oc);
    w->dmax = (unsigned*)(base + od);
    w->colA = (int*)(base + oca); w->rowT = (int*)(base + ort); w->colT = (int*)(base + oct);
  }
  return o;
}

size_t luz_matrix_bytes(int n) { return z_bytes(n, nullptr, nullptr); }

__device__ __forceinline__ ZWork z_work(const LuMat& m) {
  ZWork w;
  z_bytes(m.n, &w, (unsigned char*)m.ws);
  return w;
}

// ---------------------------------------------------------------- exponents
// Order-preserving integer of |v| 2^e: the bits of |v| with e added to the
// exponent field (biased to stay positive); 0 for zero, all ones for Inf, NaN.
__device__ __forceinline__ unsigned long long z_graded(double v, int e) {
  unsigned long long b = abs_bits(v);
  if (b == 0) return 0;
  const unsigned x = (unsigned)(b >> 52);
  if (x == 0x7FF) return ~0ull;
  if (x == 0) b = 1ull << 52;
  return b + ((unsigned long long)(e + 1024) << 52);
}
// E with |v| 2^e / 2^E < 1 for every v whose z_graded is at most g
__device__ __forceinline__ int z_scale_exp(unsigned long long g) {
  return g == 0 ? 0 : g == ~0ull ? Z_NAN : (int)(g >> 52) - 2046;
}
// exponent of the inner grading from the high word of a row's largest magnitude
__device__ __forceinline__ unsigned z_high(cd v) {
  return (unsigned)max(__double2hiint(v.x) & 0x7FFFFFFF, __double2hiint(v.y) & 0x7FFFFFFF);
}
__device__ __forceinline__ int z_grade(unsigned high) {
  const int x = (int)(high >> 20);
  return (x == 0 || x >= 0x7FF) ? 0 : x - 1023;
}

// exponent of a vector's scale as the tile's bound takes it, less that of its column of A
__device__ __forceinline__ int z_bound_exp(unsigned long long g, int E, int column) {
  return g == 0 ? Z_NONE : E >= Z_NAN ? Z_NAN : E - column;
}

// Exponents of the columns of A (0 for zero columns and those with Inf or NaN): a warp a
// column, eight columns a CTA.
__global__ void __launch_bounds__(256) z_columns_kernel(const LuMat* __restrict__ mats) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n, c = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (c >= n) return;
  const cd* col = (const cd*)mat.A + (size_t)c * n;
  unsigned mx = 0;
#pragma unroll 8
  for (int r = lane; r < n; r += 32) mx = max(mx, z_high(col[r]));
  mx = __reduce_max_sync(0xffffffffu, mx);
  if (lane == 0) z_work(mat).colA[c] = z_grade(mx);
}

// ---------------------------------------------------------------- slicing
// Grading exponents sE[k] of the K rows k0.. : from the columns [c0, c1) of the
// matrix, or from maxima already formed (dmax).  All threads.
__device__ __forceinline__ void z_grades(const cd* M, int n, int k0, int K, int c0, int c1, const unsigned* dmax,
                                         unsigned* sD, int* sE) {
  const int tid = threadIdx.x;
  if (dmax) {
    for (int k = tid; k < K; k += blockDim.x) sE[k] = z_grade(dmax[k]);
    __syncthreads();
    return;
  }
  for (int k = tid; k < K; k += blockDim.x) sD[k] = 0;
  __syncthreads();
  unsigned mx = 0;
  const int k = tid % K;
  for (int c = c0 + tid / K; c < c1; c += blockDim.x / K) mx = max(mx, z_high(M[(size_t)c * n + k0 + k]));
  if (mx) atomicMax(&sD[k], mx);
  __syncthreads();
  for (int q = tid; q < K; q += blockDim.x) sE[q] = z_grade(sD[q]);
  __syncthreads();
}

// Row operand (128-vector tiles) of the inner rows k0..k0+K.  FROM_U false: the
// rows v0.. of L times the grading; true: the columns v0.. of U divided by it.
// Grading from the columns [g0, gcap) of the matrix, or (dsel >= 0) from
// dmax[dsel..].  One CTA per tile, four threads per vector; clear: zero dmax for
// the block that begins (its U12 follows).
#define ZSL_THREADS 512
template <int K, bool FROM_U>
__global__ void __launch_bounds__(ZSL_THREADS) z_slice_rows_kernel(const LuMat* __restrict__ mats, int v0, int k0,
                                                                   int g0, int gcap, int dsel, int clear) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n, i0 = v0 + blockIdx.x * ZR, g1 = min(n, gcap);
  if (i0 >= n || g0 >= g1) return;
  const ZWork w = z_work(mat);
  const cd* M = (const cd*)mat.A;
  __shared__ unsigned long long smx[4][ZR];
  __shared__ unsigned sD[K];
  __shared__ int sE[K], sT[ZR / 32];
  if (clear && blockIdx.x == 0 && threadIdx.x < ZB) w.dmax[threadIdx.x] = 0;
  z_grades(M, n, k0, K, g0, g1, dsel >= 0 ? w.dmax + dsel : nullptr, sD, sE);
  const int r = threadIdx.x % ZR, part = threadIdx.x / ZR, i = i0 + r;
  constexpr int KP = K / 4;  // inner indices per thread
  const cd* src = FROM_U ? M + (size_t)i * n + k0 : M + (size_t)k0 * n + i;
  const size_t sk = FROM_U ? 1 : n;
  const int sg = FROM_U ? -1 : 1;
  unsigned long long g = 0;
#pragma unroll 8
  for (int q = 0; q < KP; ++q) {
    const int k = part * KP + q;
    const cd v = i < n ? src[k * sk] : C(0.0);
    g = max(g, max(z_graded(v.x, sg * sE[k]), z_graded(v.y, sg * sE[k])));
  }
  smx[part][r] = g;
  __syncthreads();
  g = max(max(smx[0][r], smx[1][r]), max(smx[2][r], smx[3][r]));
  const int E = z_scale_exp(g);
  if (part == 0) {
    w.rowE[blockIdx.x * ZR + r] = E;
    const int t = __reduce_max_sync(0xffffffffu, z_bound_exp(g, E, FROM_U && i < n ? w.colA[i] : 0));
    if ((r & 31) == 0) sT[r >> 5] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) w.rowT[blockIdx.x] = max(max(sT[0], sT[1]), max(sT[2], sT[3]));
  const int sh = E >= Z_NAN ? -8192 : 56 - E;
  for (int kg = part * KP; kg < (part + 1) * KP; kg += 8) {
    int dr[8][OZ_S], di[8][OZ_S];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const cd v = i < n ? src[(kg + c) * sk] : C(0.0);
      digits28(fixed_rn(v.x, sh + sg * sE[kg + c]), dr[c]);
      digits28(fixed_rn(v.y, sh + sg * sE[kg + c]), di[c]);
    }
    __nv_bfloat16* blk = w.Ad + ((size_t)blockIdx.x * ZKT + kg / ZK) * ZA_BLOCK + core_off(r, kg % ZK);
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
      __align__(16) __nv_bfloat16 re[8], im[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        re[c] = __float2bfloat16((float)dr[c][s]);
        im[c] = __float2bfloat16((float)di[c][s]);
      }
      *(uint4*)(blk + s * ZA_TILE) = *(const uint4*)re;
      *(uint4*)(blk + (OZ_S + s) * ZA_TILE) = *(const uint4*)im;
    }
  }
}

// Column operand (32-vector tiles): FROM_L false: the columns v0.. of U divided by
// the grading; true: the rows v0.. of L times it.  Vectors below vcap.  One CTA
// per tile; a thread holds 8 inner indices of one vector.
template <int K, bool FROM_L>
__global__ void __launch_bounds__(256) z_slice_cols_kernel(const LuMat* __restrict__ mats, int v0, int vcap, int k0,
                                                           int g0, int gcap, int dsel) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n, j0 = v0 + blockIdx.x * ZC, v1 = min(n, vcap), g1 = min(n, gcap);
  if (j0 >= v1 || g0 >= g1) return;
  const ZWork w = z_work(mat);
  const cd* M = (const cd*)mat.A;
  __shared__ unsigned sD[K];
  __shared__ int sE[K], sT;
  if (threadIdx.x == 0) sT = Z_NONE;
  z_grades(M, n, k0, K, g0, g1, dsel >= 0 ? w.dmax + dsel : nullptr, sD, sE);
  constexpr int G = K / 8;  // threads per vector
  const int sg = FROM_L ? 1 : -1;
  for (int it = threadIdx.x; it < ZC * G; it += 256) {  // whole warps: ZC G is a multiple of 32
    const int jj = it / G, kg = (it % G) * 8, j = j0 + jj;
    cd v[8];
    unsigned long long g = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      v[c] = j < v1 ? (FROM_L ? M[(size_t)(k0 + kg + c) * n + j] : M[(size_t)j * n + k0 + kg + c]) : C(0.0);
      g = max(g, max(z_graded(v[c].x, sg * sE[kg + c]), z_graded(v[c].y, sg * sE[kg + c])));
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) g = max(g, __shfl_xor_sync(0xffffffffu, g, o));
    const int E = z_scale_exp(g);
    if (kg == 0) {
      w.colE[blockIdx.x * ZC + jj] = E;
      atomicMax(&sT, z_bound_exp(g, E, !FROM_L && j < v1 ? w.colA[j] : 0));
    }
    const int sh = E >= Z_NAN ? -8192 : 56 - E;
    int dr[8][OZ_S], di[8][OZ_S];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      digits28(fixed_rn(v[c].x, sh + sg * sE[kg + c]), dr[c]);
      digits28(fixed_rn(v[c].y, sh + sg * sE[kg + c]), di[c]);
    }
    __nv_bfloat16* blk = w.Bd + ((size_t)blockIdx.x * ZKT + kg / ZK) * ZB_BLOCK + core_off(jj, kg % ZK);
#pragma unroll
    for (int s = 0; s < OZ_S; ++s) {
      __align__(16) __nv_bfloat16 re[8], im[8], nim[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        re[c] = __float2bfloat16((float)dr[c][s]);
        im[c] = __float2bfloat16((float)di[c][s]);
        nim[c] = __float2bfloat16((float)-di[c][s]);
      }
      *(uint4*)(blk + (2 * s) * ZB_TILE) = *(const uint4*)re;
      *(uint4*)(blk + (2 * s + 1) * ZB_TILE) = *(const uint4*)im;
      *(uint4*)(blk + (2 * OZ_S + 2 * s) * ZB_TILE) = *(const uint4*)nim;
      *(uint4*)(blk + (2 * OZ_S + 2 * s + 1) * ZB_TILE) = *(const uint4*)re;
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) w.colT[blockIdx.x] = sT;
}

// Rows k0..k0+LU_NB of U in the columns [c0, ccap): unit-lower triangular solve,
// 32 columns per CTA; dsel >= 0: also the rows' largest magnitudes (high words) into
// dmax[dsel..].  The products with the rows above are summed before they are
// subtracted: four FP64 operations a term and one rounding of the result's
// size per row.  Four warps, one per FP64 pipe of the SM, share a column (warp
// w holds the sums of rows w, w + 4, ..): with one warp per 32 columns its own
// pipe alone took 64 clocks an operation, 89 us per launch (n = 1250, 9 matrices).
__global__ void __launch_bounds__(128) z_trsm_kernel(const LuMat* __restrict__ mats, int k0, int c0, int ccap, int dsel) {
  const LuMat mat = mats[blockIdx.y];
  const int n = mat.n, b0 = c0 + blockIdx.x * 32, c1 = min(n, ccap), lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (b0 >= c1) return;
  cd* M = (cd*)mat.A;
  __shared__ cd L[LU_NB][LU_NB + 1], B[LU_NB][LU_NB + 1];  // B[column][row]
  for (int c = w; c < LU_NB; c += 4) {
    L[lane][c] = M[(size_t)(k0 + c) * n + k0 + lane];
    B[c][lane] = b0 + c < c1 ? M[(size_t)(b0 + c) * n + k0 + lane] : C(0.0);
  }
  __syncthreads();
  cd acc[LU_NB / 4];
#pragma unroll
  for (int q = 0; q < LU_NB / 4; ++q) acc[q] = C(0.0);
#pragma unroll
  for (int k = 0; k < LU_NB; ++k) {
    if (w == (k & 3)) B[lane][k] = B[lane][k] - acc[k >> 2];
    __syncthreads();
    const cd x = B[lane][k];
#pragma unroll
    for (int q = 0; q < LU_NB / 4; ++q) {
      const int r = w + 4 * q;
      if (4 * q + 3 > k && r > k) acc[q] = fma(L[r][k], x, acc[q]);
    }
    if (dsel >= 0 && w == (k & 3)) {
      const unsigned mx = __reduce_max_sync(0xffffffffu, z_high(x));
      if (lane == 0 && mx) atomicMax(&z_work(mat).dmax[dsel + k], mx);
    }
  }
  __syncthreads();
  for (int c = w; c < LU_NB; c += 4)
    if (b0 + c < c1) M[(size_t)(b0 + c) * n + k0 + lane] = B[c][lane];
}

// ---------------------------------------------------------------- product
// C[r0 + i, c0 + j] -= sum_k A_ik B_kj over the tiles (128 x 32) of every matrix
// (columns below ccap; SWAP: tile rows are matrix columns),
// persistent, one CTA per SM.  Warps 0-15 drain (warp w: tensor-memory
// lanes 32 (w & 3).., columns 8 (w >> 2)..), warp 16 copies k-tiles through a ring
// of two stages, warp 17 issues MMAs.  The accumulators (8 levels x [Re | Im] x
// 32) fill tensor memory, so a tile is handed over in two halves: the last
// k-tile's products of levels 0-3 are issued and committed before those of
// levels 4-7, and the next tile may start on the half already drained.
// Every wait is bounded: a role that gives up sets the CTA's failure flag (and
// *err), the others stop at their next wait, and before the CTA exits the
// copies in flight land and the MMAs complete.
// Tiles that the digits would not keep (Z_SAFE) are no work for copies and MMAs; the drain
// warps form them from L and U (inner rows k0 ..) in FP64.

// Row i of such a tile, its columns j0 .. j0 + nc - 1.
template <bool SWAP>
__device__ __noinline__ void z_tile_fp64(cd* M, int n, int k0, int K, int i, int j0, int nc) {
  cd acc[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) acc[c] = C(0.0);
  for (int k = k0; k < k0 + K; ++k) {
    const cd a = SWAP ? M[(size_t)i * n + k] : M[(size_t)k * n + i];
#pragma unroll
    for (int c = 0; c < 8; ++c)
      if (c < nc) acc[c] = fma(a, SWAP ? M[(size_t)k * n + j0 + c] : M[(size_t)(j0 + c) * n + k], acc[c]);
  }
#pragma unroll
  for (int c = 0; c < 8; ++c)
    if (c < nc) {
      cd* o = SWAP ? M + (size_t)i * n + j0 + c : M + (size_t)(j0 + c) * n + i;
      *o = *o - acc[c];
    }
}

template <bool SWAP>
__global__ void __launch_bounds__(Z_THREADS, 1) z_product_kernel(const LuMat* __restrict__ mats, int k0, int r0, int c0,
                                                                 int ccap, int nkt, int nrt, int nct, int count,
                                                                 int* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[Z_NST], empty[Z_NST], tfull[2], tempty[2], mdone;
  __shared__ uint32_t tmem_base;
  __shared__ int s_fail;
  volatile int* fail = &s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long per = (long long)nrt * nct, total = per * count;
  auto tile_of = [&](long long t, int& z, int& x, int& y) -> bool {
    z = (int)(t / per);
    const long long r = t - (long long)z * per;
    y = (int)(r / nrt);
    x = (int)(r - (long long)y * nrt);
    const int n = mats[z].n;
    return r0 + x * ZR < n && c0 + y * ZC < min(n, ccap);
  };
  auto kept = [](const ZWork& w, int x, int y) { return w.rowT[x] + w.colT[y] <= Z_SAFE; };
  if (warp == 0) tc::tmem_alloc(&tmem_base, 512);
  if (tid == 32) {
    s_fail = 0;
    for (int b = 0; b < Z_NST; ++b) { tc::mbar_init(&full[b], 1); tc::mbar_init(&empty[b], 1); }
    for (int b = 0; b < 2; ++b) { tc::mbar_init(&tfull[b], 1); tc::mbar_init(&tempty[b], Z_DRAIN); }
    tc::mbar_init(&mdone, 1);
    tc::mbar_fence_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t tmem = tmem_base;
  int issued = 0;
  if (warp == Z_DRAIN) {
    if (lane == 0) {
      int q = 0;
      for (long long t = blockIdx.x; t < total && !*fail; t += gridDim.x) {
        int z, x, y;
        if (!tile_of(t, z, x, y)) continue;
        const ZWork w = z_work(mats[z]);
        if (!kept(w, x, y)) continue;
        const __nv_bfloat16* As = w.Ad + (size_t)x * ZKT * ZA_BLOCK;
        const __nv_bfloat16* Bs = w.Bd + (size_t)y * ZKT * ZB_BLOCK;
        for (int kt = 0; kt < nkt; ++kt, ++q) {
          const int st = q % Z_NST;
          if (q >= Z_NST && !tc::mbar_wait(&empty[st], ((q / Z_NST) - 1) & 1)) { *fail = 1; break; }
          unsigned char* base = smem + (size_t)st * Z_STAGE;
          tc::mbar_expect_tx(&full[st], Z_STAGE);
          tc::bulk_g2s(base, As + (size_t)kt * ZA_BLOCK, ZA_BLOCK * 2, &full[st]);
          tc::bulk_g2s(base + ZA_BLOCK * 2, Bs + (size_t)kt * ZB_BLOCK, ZB_BLOCK * 2, &full[st]);
          issued = q + 1;
        }
      }
    }
  } else if (warp == Z_DRAIN + 1) {
    if (lane == 0) {
      int q = 0, k = 0;
      for (long long t = blockIdx.x; t < total && !*fail; t += gridDim.x) {
        int z, x, y;
        if (!tile_of(t, z, x, y) || !kept(z_work(mats[z]), x, y)) continue;
        for (int kt = 0; kt < nkt && !*fail; ++kt, ++q) {
          const int st = q % Z_NST;
          if (!tc::mbar_wait(&full[st], (q / Z_NST) & 1)) { *fail = 1; break; }
          unsigned char* base = smem + (size_t)st * Z_STAGE;
          const uint64_t a0 = tc::desc_noswizzle(tc::smem_u32(base), 128, 256);
          const uint64_t b0 = tc::desc_noswizzle(tc::smem_u32(base + ZA_BLOCK * 2), 128, 256);
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            if (kt == 0 && k > 0 && !tc::mbar_wait(&tempty[half], (k - 1) & 1)) { *fail = 1; break; }
            tc::fence_after();
#pragma unroll
            for (int sd = 0; sd < 4 * half + 4; ++sd) {  // digit sd of L times the digits td, td + 1, ..: levels l, l + 1, ..
              const int l = sd > 4 * half ? sd : 4 * half, td = l - sd;
              const uint32_t idesc = tc::idesc_bf16_f32(ZR, 2 * ZC * (4 * half + 4 - l)), acc = tmem + (uint32_t)(l * 2 * ZC);
              const uint64_t are = a0 + (uint64_t)(sd * (ZA_TILE * 2 / 16));
              const uint64_t aim = a0 + (uint64_t)((OZ_S + sd) * (ZA_TILE * 2 / 16));
              const uint64_t bri = b0 + (uint64_t)(2 * td * (ZB_TILE * 2 / 16));
              tc::mma_bf16(acc, are, bri, idesc, (kt == 0 && sd == 0) ? 0u : 1u);
              tc::mma_bf16(acc, aim, bri + (uint64_t)(2 * OZ_S * (ZB_TILE * 2 / 16)), idesc, 1u);
            }
            if (kt == nkt - 1) tc::commit(&tfull[half]);
          }
          if (*fail) break;
          tc::commit(&empty[st]);
        }
        ++k;
      }
      tc::commit(&mdone);
      if (!tc::mbar_wait(&mdone, 0)) *fail = 1;
    }
  } else {
    int k = 0;
    for (long long t = blockIdx.x; t < total; t += gridDim.x) {
      int z, x, y;
      if (!tile_of(t, z, x, y)) continue;
      const LuMat mat = mats[z];
      const ZWork w = z_work(mat);
      const int n = mat.n, i = r0 + x * ZR + (warp & 3) * 32 + lane, jt = y * ZC + (warp >> 2) * 8;
      const int nc = i < n ? min(8, min(n, ccap) - c0 - jt) : 0;  // columns of this thread's row
      cd* M = SWAP ? (cd*)mat.A + (size_t)i * n + c0 + jt : (cd*)mat.A + (size_t)(c0 + jt) * n + i;
      const size_t sc = SWAP ? 1 : n;
      if (!kept(w, x, y)) {
        if (nc > 0) z_tile_fp64<SWAP>((cd*)mat.A, n, k0, nkt * ZK, i, c0 + jt, nc);
        continue;
      }
      const int Er = w.rowE[x * ZR + (warp & 3) * 32 + lane] - 54;
      if (!tc::mbar_wait(&tfull[0], k & 1)) { *fail = 1; break; }
      tc::fence_after();
      const uint32_t tw = tmem + (uint32_t)((warp >> 2) * 8) + ((uint32_t)((warp & 3) * 32) << 16);
      // levels 0-3: hi = sum acc_l 2^{7 (3 - l)}, pairs joined in 32 bits
      long long hi[2][8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[4][8];
        tc::tmem_ld8x4(tw + h * ZC, tw + 2 * ZC + h * ZC, tw + 4 * ZC + h * ZC, tw + 6 * ZC + h * ZC, v);
#pragma unroll
        for (int c = 0; c < 8; ++c)
          hi[h][c] = (long long)(__float2int_rn(v[0][c]) * 128 + __float2int_rn(v[1][c])) * 16384 +
                     (__float2int_rn(v[2][c]) * 128 + __float2int_rn(v[3][c]));
      }
      tc::fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&tempty[0]);
      cd cv[8];
#pragma unroll
      for (int c = 0; c < 8; ++c)  // C while the products of levels 4-7 finish
        cv[c] = c < nc ? M[c * sc] : C(0.0);
      if (!tc::mbar_wait(&tfull[1], k & 1)) { *fail = 1; break; }
      tc::fence_after();
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float v[4][8];
        tc::tmem_ld8x4(tw + 8 * ZC + h * ZC, tw + 10 * ZC + h * ZC, tw + 12 * ZC + h * ZC, tw + 14 * ZC + h * ZC, v);
        if (h == 1) {
          tc::fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive(&tempty[1]);
        }
        // hi in units of 2^-35, lo of 2^-63: V in units of 2^-54 (below 2^63)
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const long long lo = (long long)(__float2int_rn(v[0][c]) * 128 + __float2int_rn(v[1][c])) * 16384 +
                               (__float2int_rn(v[2][c]) * 128 + __float2int_rn(v[3][c]));
          const long long V = hi[h][c] * 524288 + ((lo + 256) >> 9);
          const int E = Er + w.colE[jt + c];
          const double d = E >= Z_NAN / 2 ? nan("") : fixed_to_double(V, E);
          if (h == 0) cv[c].x -= d;
          else cv[c].y -= d;
        }
      }
#pragma unroll
      for (int c = 0; c < 8; ++c)
        if (c < nc) M[c * sc] = cv[c];
      ++k;
    }
  }
  __syncthreads();
  if (*fail) {
    if (tid == 0 && err) atomicExch(err, 1);
    if (warp == Z_DRAIN && lane == 0) {
      for (int st = 0; st < Z_NST; ++st) {
        const int last = issued - 1 - ((issued - 1 - st) % Z_NST + Z_NST) % Z_NST;  // newest k-tile issued into st
        if (last >= 0) tc::mbar_wait(&full[st], (last / Z_NST) & 1, 1 << 20);
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------- launches
static int z_sms() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

template <bool SWAP>
static void z_product(const LuMat* d, int k0, int r0, int rows, int c0, int ccap, int cols, int K, int count, int* err,
                      cudaStream_t s) {
  const int nrt = z_tiles(rows, ZR), nct = z_tiles(cols, ZC);
  cudaFuncSetAttribute(z_product_kernel<SWAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, Z_NST * Z_STAGE);
  const int grid = (int)std::min<long long>((long long)nrt * nct * count, z_sms());
  z_product_kernel<SWAP><<<grid, Z_THREADS, Z_NST * Z_STAGE, s>>>(d, k0, r0, c0, ccap, K / ZK, nrt, nct, count, err);
}

void luz_begin(const LuMat* d, int nmax, int count, cudaStream_t s) {
  z_columns_kernel<<<dim3(z_tiles(nmax, 8), count), 256, 0, s>>>(d);
}

void luz_panel_rows(const LuMat* d, int K0, int k0, int cols, int count, cudaStream_t s) {
  z_trsm_kernel<<<dim3(z_tiles(cols, 32), count), 128, 0, s>>>(d, k0, k0 + LU_NB, K0 + ZB, -1);
}

int luz_panel_update(const LuMat* d, int K0, int k0, int nmax, int count, int* err, cudaStream_t s) {
  const int r0 = k0 + LU_NB, ccap = K0 + ZB, cols = std::min(ccap, nmax) - r0, rows = nmax - r0;
  z_slice_rows_kernel<LU_NB, false><<<dim3(z_tiles(rows, ZR), count), ZSL_THREADS, 0, s>>>(d, r0, k0, r0, ccap, -1,
                                                                                           k0 == K0);
  z_slice_cols_kernel<LU_NB, false><<<dim3(z_tiles(cols, ZC), count), 256, 0, s>>>(d, r0, ccap, k0, r0, ccap, -1);
  z_product<false>(d, k0, r0, rows, r0, ccap, cols, LU_NB, count, err, s);
  return 3;
}

int luz_block_update(const LuMat* d, int K0, int nmax, int count, int* err, cudaStream_t s) {
  const int r0 = K0 + ZB, rest = nmax - r0, cap = 1 << 30;
  int launches = 0;
  for (int k0 = K0; k0 < r0; k0 += LU_NB) {
    z_trsm_kernel<<<dim3(z_tiles(rest, 32), count), 128, 0, s>>>(d, k0, r0, cap, k0 - K0);
    ++launches;
    const int v0 = k0 + LU_NB, brows = r0 - v0;
    if (brows <= 0) break;
    z_slice_rows_kernel<LU_NB, true><<<dim3(z_tiles(rest, ZR), count), ZSL_THREADS, 0, s>>>(d, r0, k0, r0, cap,
                                                                                            k0 - K0, 0);
    z_slice_cols_kernel<LU_NB, true><<<dim3(z_tiles(brows, ZC), count), 256, 0, s>>>(d, v0, r0, k0, r0, cap, k0 - K0);
    z_product<true>(d, k0, r0, rest, v0, r0, brows, LU_NB, count, err, s);
    launches += 3;
  }
  z_slice_rows_kernel<ZB, false><<<dim3(z_tiles(rest, ZR), count), ZSL_THREADS, 0, s>>>(d, r0, K0, r0, cap, 0, 0);
  z_slice_cols_kernel<ZB, false><<<dim3(z_tiles(rest, ZC), count), 256, 0, s>>>(d, r0, cap, K0, r0, cap, 0);
  z_product<false>(d, K0, r0, rest, r0, cap, rest, ZB, count, err, s);
  return launches + 3;
}
