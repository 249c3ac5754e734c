// Triangular solves with the LU factors of all modes, for right-hand sides of
// modes -M..M (n is a multiple of 64: 16 nodes of 4 unknowns per panel).
//
// One launch per 64-column block of the factor and sweep: with the block's part
// x_k of the solution known, every CTA takes 128 rows (of one mode and a group
// of VT vectors) and subtracts L_ik x_k, and the CTA that owns the next block's
// rows then solves its 64 x 64 triangle and leaves x_{k+1} for the next launch.
// So the factor is read once per group by all SMs at once; one CTA per mode and
// group walking the whole factor (the form this replaces) left it to as many SMs
// as there are modes, each waiting for its own chain of blocks.
// Three solves: N = 1024, M = 128, 4 vectors per mode (complex64) 29.3 -> 17.6 ms;
// one complex128 solve, N = 320, M = 64, 8 vectors 13.0 -> 9.6 ms (FP64 pipe).
//
// Groups of 4 or 8 vectors are bound by the factor's bytes (complex64) or the
// FP64 pipe (complex128): the tile goes straight to registers, 16 bytes a load,
// four (two) column groups per tile added in shared memory.  Groups of 16, 32 or
// 64 (complex64) form the products on the tensor cores (solve_tc_kernel).
//
// x holds the vectors in FP64; the sums over a block's 64 columns and the
// triangles run in the factor's precision.
#include <algorithm>
#include <type_traits>
#include "cplx.cuh"
#include "lu.cuh"
#include "smem.cuh"
#include "split3.cuh"
#include "tc.cuh"

#define SB 64    // columns of a block
#define SRT 128  // rows of a tile

namespace {

// job: (right-hand side, sign); sign - is mode -m, solved with A_{-m} = D_r A_m D_c
__device__ __forceinline__ void job_of(int m, int M, int nrhs, int job, int* q, int* ridx, bool* neg) {
  *ridx = job % nrhs;
  *neg = job >= nrhs;
  *q = *neg ? (M - m) : (M + m);
}

template <class T> __device__ __forceinline__ T conv(cd a);
template <> __device__ __forceinline__ cd conv<cd>(cd a) { return a; }
template <> __device__ __forceinline__ cf conv<cf>(cd a) { return to_cf(a); }
// FP32 -> FP64 on the integer pipe (normal numbers and zero; the call keeps the
// conversion of the others out of the common path): an FP64 conversion costs as
// much as the FP64 subtraction that follows it.
__device__ __noinline__ double widen_other(float f) { return (double)f; }
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f), a = u & 0x7FFFFFFFu;
  if (a - 0x00800000u >= 0x7F000000u && a != 0u) return widen_other(f);
  const unsigned hi = (u & 0x80000000u) | (a ? (a >> 3) + (896u << 20) : 0u);
  return __hiloint2double((int)hi, (int)(u << 29));
}
// Vectors of the library's own buffers are 16-byte aligned; a caller's need not be.
template <bool OWN> __device__ __forceinline__ cd load_x(const cd* p) {
  if (OWN) { const double2 v = *(const double2*)p; return cd{v.x, v.y}; }
  return *p;
}
template <bool OWN> __device__ __forceinline__ void store_x(cd* p, cd v) {
  if (OWN) *(double2*)p = make_double2(v.x, v.y);
  else *p = v;
}
__device__ __forceinline__ cd wide(cf a) { return cd{widen(a.x), widen(a.y)}; }
__device__ __forceinline__ cd wide(cd a) { return a; }

template <class T> __device__ __forceinline__ T shfl_c(T v, int src) {
  T r;
  r.x = __shfl_sync(0xffffffffu, v.x, src);
  r.y = __shfl_sync(0xffffffffu, v.y, src);
  return r;
}

// perm[m][r]: the row interchanges of mode m (LAPACK order) composed, (P b)[r] =
// b[perm[r]].  The 32 interchanges of a panel move at most 64 rows: 32 warps form
// the moves of 32 panels at a time, then warp 0 applies the panels in order.
__global__ void __launch_bounds__(1024) perm_kernel(const int* __restrict__ piv, int n, int* __restrict__ perm_out) {
  extern __shared__ int perm[];  // [n]
  __shared__ int pos[32][64], src[32][64], slot[32][32];
  const int* pv = piv + (size_t)blockIdx.x * n;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int r = threadIdx.x; r < n; r += blockDim.x) perm[r] = r;
  for (int b0 = 0; b0 < n; b0 += 1024) {
    __syncthreads();
    const int k0 = b0 + 32 * warp;
    if (k0 < n) {  // n is a multiple of 32
      const int p = pv[k0 + lane];
      const unsigned same = __match_any_sync(0xffffffffu, p);
      const bool below = p >= k0 + 32, first = below && (__ffs(same) - 1 == lane);
      pos[warp][lane] = src[warp][lane] = k0 + lane;
      pos[warp][32 + lane] = src[warp][32 + lane] = first ? p : -1;
      slot[warp][lane] = below ? 32 + __ffs(same) - 1 : p - k0;
      __syncwarp();
      if (lane == 0)
        for (int k = 0; k < 32; ++k) {
          const int s2 = slot[warp][k];
          if (s2 != k) { const int t = src[warp][k]; src[warp][k] = src[warp][s2]; src[warp][s2] = t; }
        }
    }
    __syncthreads();
    if (warp == 0)
      for (int w = 0; w < 32 && b0 + 32 * w < n; ++w) {
        const int d0 = pos[w][lane], d1 = pos[w][32 + lane], s0 = src[w][lane], s1 = src[w][32 + lane];
        const int v0 = perm[s0], v1 = d1 >= 0 ? perm[s1] : 0;
        __syncwarp();
        perm[d0] = v0;
        if (d1 >= 0) perm[d1] = v1;
        __syncwarp();
      }
  }
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += blockDim.x) perm_out[(size_t)blockIdx.x * n + r] = perm[r];
}

// x = the permuted right-hand sides: scaled (PHYS: by the sqrt weight per node)
// and reflected for -m.
template <bool PHYS>
__global__ void __launch_bounds__(256) solve_init_kernel(int n, int M, int nrhs, const int* __restrict__ perm,
                                                         const double* __restrict__ sw, const cd* __restrict__ rhs,
                                                         cd* __restrict__ x) {
  const int m = blockIdx.y, njobs = m == 0 ? nrhs : 2 * nrhs;
  const int r = blockIdx.x * 256 + threadIdx.x;
  if (r >= n) return;
  const int src = perm[(size_t)m * n + r];
  const double s = PHYS ? sw[src >> 2] : 1.0;
  const bool flip = (src & 3) == 0 || (src & 3) == 3;
  for (int job = blockIdx.z; job < njobs; job += gridDim.z) {
    int q, ri; bool neg;
    job_of(m, M, nrhs, job, &q, &ri, &neg);
    const size_t o = ((size_t)q * nrhs + ri) * n;
    x[o + r] = ((neg && flip) ? -s : s) * rhs[o + src];
  }
}

template <class TF> struct SolveArgs {
  const TF* LU;
  TF* xb;            // block solutions: [parity][mode][group][SB][VT]
  const double* sw;
  cd* x;
  int n, M, nrhs, groups;
};

template <class TF, int VT> struct SolveShape {
  static constexpr int CG = std::is_same<TF, cf>::value ? 4 : 2;  // column groups of a tile
  static constexpr int XS = SB * VT * (int)sizeof(TF);             // block solution
  static constexpr int DIAG = (SB * SB + SB) * (int)sizeof(TF);    // triangle and reciprocals
  static constexpr int TILE = CG * VT * SRT * (int)sizeof(TF);     // partial sums
  // complex64 (latency counts): the triangle has its own space and is fetched at the
  // start; else it takes the partial sums'
  static constexpr bool EARLY = std::is_same<TF, cf>::value;
  static constexpr int SMEM = 2 * XS + (EARLY ? TILE + DIAG : TILE > DIAG ? TILE : DIAG) + VT * 8;
};

// The next block's triangle, column-major (factors are the library's own: columns
// of a multiple of 64 entries).
template <class TF> __device__ __forceinline__ void load_triangle(TF* D, const TF* L, int n, int kc) {
  const TF* Fd = L + (size_t)kc * SB * n + kc * SB;
  constexpr int Q = 16 / sizeof(TF);
  for (int e = threadIdx.x; e < SB * SB / Q; e += 256) {
    const int c = e / (SB / Q), r = (e % (SB / Q)) * Q;
    *(uint4*)(D + c * SB + r) = *(const uint4*)(Fd + (size_t)c * n + r);
  }
}

// The triangle of a block for the vectors j0 .. j0 + JC - 1 by one warp: lane holds
// rows lane and lane + 32; products are summed apart (s) and subtracted once.
template <class TF, int VT, int JC, bool FWD>
__device__ __forceinline__ void solve_triangle(const TF* D, const TF* inv, const TF* Bs, int j0, TF (&b)[2][JC]) {
  const int lane = threadIdx.x & 31;
  TF s[2][JC];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < JC; ++j) {
      b[h][j] = Bs[(lane + 32 * h) * VT + j0 + j];
      s[h][j] = czero<TF>();
    }
#pragma unroll
  for (int hh = 0; hh < 2; ++hh) {
    const int h = FWD ? hh : 1 - hh;  // half whose columns are eliminated
    for (int cc = 0; cc < 32; ++cc) {
      const int cl = FWD ? cc : 31 - cc, c = cl + 32 * h;
      TF xc[JC];
#pragma unroll
      for (int j = 0; j < JC; ++j) {
        TF v = b[h][j] - s[h][j];
        if (!FWD) v = v * inv[c];
        xc[j] = shfl_c(v, cl);
        if (lane == cl) { b[h][j] = xc[j]; s[h][j] = czero<TF>(); }
      }
      const bool below = FWD ? lane > cl : lane < cl;
      if (below) {
        const TF l = D[c * SB + lane + 32 * h];
#pragma unroll
        for (int j = 0; j < JC; ++j) s[h][j] = fma(l, xc[j], s[h][j]);
      }
      if (hh == 0) {  // the other half lies wholly beyond
        const TF l = D[c * SB + lane + 32 * (1 - h)];
#pragma unroll
        for (int j = 0; j < JC; ++j) s[1 - h][j] = fma(l, xc[j], s[1 - h][j]);
      }
    }
  }
}

// One block step (see above); first: no update, only the first block's triangle.
// The backward sweep leaves the finished unknowns: reflected for -m and (PHYS)
// divided by the sqrt weights.
template <class TF, int VT, bool FWD, bool PHYS>
__global__ void __launch_bounds__(256, 2) solve_step_kernel(SolveArgs<TF> a, int k, int first) {
  using S = SolveShape<TF, VT>;
  extern __shared__ __align__(16) unsigned char sraw[];
  TF* xs = (TF*)sraw;                    // [SB][VT] solution of block k
  TF* Bs = (TF*)(sraw + S::XS);          // [SB][VT] right-hand side of the next block
  TF* T = (TF*)(sraw + 2 * S::XS);       // tile or partial sums
  TF* D = S::EARLY ? (TF*)(sraw + 2 * S::XS + S::TILE) : T;  // triangle of the next block, column-major
  TF* inv = D + SB * SB;                 // reciprocals of its diagonal
  size_t* voff = (size_t*)(sraw + S::SMEM - VT * 8);  // [VT] the vectors in x
  const int n = a.n, m = blockIdx.y, g = blockIdx.z, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int njobs = m == 0 ? a.nrhs : 2 * a.nrhs, job0 = g * VT;
  if (job0 >= njobs) return;
  const int G = min(VT, njobs - job0), nblk = n / SB;
  const TF* L = a.LU + (size_t)m * n * n;
  const int kc = first ? (FWD ? 0 : nblk - 1) : (FWD ? k + 1 : k - 1);  // the next block
  const bool crit = blockIdx.x == 0;
  int r0, rows;
  if (first) { r0 = kc * SB; rows = SB; }
  else if (FWD) { r0 = (k + 1) * SB + SRT * blockIdx.x; rows = min(SRT, n - r0); }
  else { const int e = k * SB - SRT * blockIdx.x; r0 = max(0, e - SRT); rows = e - r0; }
  const int coff = FWD ? 0 : rows - SB;  // the next block's rows within the first tile
  auto slot = [&](int kb) { return a.xb + (((size_t)(kb & 1) * (a.M + 1) + m) * a.groups + g) * (SB * VT); };
  auto in_next = [&](int row) { return crit && row >= coff && row < coff + SB; };
  auto copy16 = [&](TF* dst, const TF* src, int bytes) {  // 16-byte aligned, contiguous
    for (int e = tid; e < bytes / 16; e += 256) ((uint4*)dst)[e] = ((const uint4*)src)[e];
  };
  if (tid < VT) {
    int q, ri; bool neg;
    job_of(m, a.M, a.nrhs, job0 + min(tid, G - 1), &q, &ri, &neg);
    voff[tid] = ((size_t)q * a.nrhs + ri) * n;
  }
  const TF* F = L + (size_t)k * SB * n + r0;
  if (first) {
    __syncthreads();
    for (int e = tid; e < SB * VT; e += 256) {
      const int row = e % SB, v = e / SB;
      Bs[row * VT + v] = v < G ? conv<TF>(a.x[voff[v] + r0 + row]) : czero<TF>();
    }
    if (S::EARLY) load_triangle(D, L, n, kc);
  } else {
    const TF* xk = slot(k);
    constexpr int NE = SRT * VT / 256;  // elements per thread of the tile's result
    cd xv0[NE];
    auto fetch_x = [&] {
#pragma unroll
      for (int q = 0; q < NE; ++q) {
        const int e = tid + 256 * q, row = e % SRT, v = e / SRT;
        xv0[q] = (row < rows && v < G) ? load_x<!PHYS>(a.x + voff[v] + r0 + row) : C(0.0);
      }
    };
    if constexpr (std::is_same<TF, cf>::value) {  // thread: two rows, 16 columns
      const int ra = 2 * (tid & 63), cg = tid >> 6;
      float4 l[SB / 4];
      if (ra < rows) {
#pragma unroll
        for (int c = 0; c < SB / 4; ++c) l[c] = __ldg((const float4*)(F + (size_t)(cg * (SB / 4) + c) * n + ra));
      }
      copy16(xs, xk, S::XS);
      if (crit) load_triangle(D, L, n, kc);
      __syncthreads();
      fetch_x();
      TF acc[2][VT];
#pragma unroll
      for (int v = 0; v < VT; ++v) acc[0][v] = acc[1][v] = czero<TF>();
      if (ra < rows) {
#pragma unroll
        for (int c = 0; c < SB / 4; ++c)
#pragma unroll
          for (int v = 0; v < VT; v += 2) {
            const float4 x2 = *(const float4*)(xs + (cg * (SB / 4) + c) * VT + v);
            acc[0][v] = fma(CF(l[c].x, l[c].y), CF(x2.x, x2.y), acc[0][v]);
            acc[1][v] = fma(CF(l[c].z, l[c].w), CF(x2.x, x2.y), acc[1][v]);
            acc[0][v + 1] = fma(CF(l[c].x, l[c].y), CF(x2.z, x2.w), acc[0][v + 1]);
            acc[1][v + 1] = fma(CF(l[c].z, l[c].w), CF(x2.z, x2.w), acc[1][v + 1]);
          }
      }
#pragma unroll
      for (int v = 0; v < VT; ++v)
        *(float4*)(T + (cg * VT + v) * SRT + ra) = make_float4(acc[0][v].x, acc[0][v].y, acc[1][v].x, acc[1][v].y);
    } else {  // thread: one row, 32 columns
      copy16(xs, xk, S::XS);
      __syncthreads();
      fetch_x();
      const int ra = tid & 127, cg = tid >> 7;
      TF acc[VT];
#pragma unroll
      for (int v = 0; v < VT; ++v) acc[v] = czero<TF>();
      if (ra < rows) {
#pragma unroll 8
        for (int c = 0; c < SB / 2; ++c) {
          const TF l = F[(size_t)(cg * (SB / 2) + c) * n + ra];
#pragma unroll
          for (int v = 0; v < VT; ++v) acc[v] = fma(l, xs[(cg * (SB / 2) + c) * VT + v], acc[v]);
        }
      }
#pragma unroll
      for (int v = 0; v < VT; ++v) T[(cg * VT + v) * SRT + ra] = acc[v];
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < NE; ++q) {
      const int e = tid + 256 * q, row = e % SRT, v = e / SRT;
      if (row >= rows) continue;
      TF sum = T[v * SRT + row];
#pragma unroll
      for (int cg = 1; cg < S::CG; ++cg) sum = sum + T[(cg * VT + v) * SRT + row];
      const cd val = xv0[q] - wide(sum);
      if (in_next(row)) Bs[(row - coff) * VT + v] = conv<TF>(val);
      else if (v < G) store_x<!PHYS>(a.x + voff[v] + r0 + row, val);
    }
    __syncthreads();
  }
  if (!crit) return;
  if (!S::EARLY) load_triangle(D, L, n, kc);
  __syncthreads();
  if (!FWD) {
    if (tid < SB) inv[tid] = cone<TF>() / D[tid * SB + tid];
    __syncthreads();
  }
  constexpr int JC = VT >= 8 ? VT / 8 : 1;  // vectors of a warp
  const int j0 = warp * JC;
  if (j0 >= VT) return;
  TF b[2][JC];
  solve_triangle<TF, VT, JC, FWD>(D, inv, Bs, j0, b);
  TF* xo = slot(kc);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < JC; ++j) {
      const int r = lane + 32 * h, v = j0 + j;
      xo[r * VT + v] = b[h][j];
      if (v >= G) continue;
      cd val = wide(b[h][j]);
      if (!FWD) {
        int q, ri; bool neg;
        job_of(m, a.M, a.nrhs, job0 + v, &q, &ri, &neg);
        const int row = kc * SB + r;
        const bool flip = neg && ((row & 3) == 1 || (row & 3) == 2);
        if (PHYS) val = ((flip ? -1.0 : 1.0) / a.sw[row >> 2]) * val;
        else if (flip) val = -val;
      }
      a.x[voff[v] + kc * SB + r] = val;
    }
}

// ---- complex64, groups of VT = 16, 32 or 64 vectors: products on the tensor cores
//
// A CTA's 128 rows of the update are the product of a 128 x 64 tile of the factor
// with the block solution of VT vectors, in two chunks of 32 columns. Every FP32
// value is split exactly into three BF16 pieces; the six piece products that carry
// FP32 precision are accumulated in tensor memory, the leading one apart from the
// five corrections, as in the complex64 factorization's update. The solution's
// pieces come as an image of rows (-Im, Re, Im) per piece, so that Re L times
// (Re, Im) and Im L times (-Im, Re), each one instruction of 2 VT columns, add to
// the same accumulators (Re, Im). The factor's pieces are formed by the CTA from the
// FP32 tile; the block solution's once, by the CTA that solves the triangle.
//
// What bounds it: the vectors' FP64 values are read and written once a block step,
// by whose bytes the step is bound; the CUDA-core form this replaces was bound by
// FP32 multiply-adds. Three solves of 192 vectors per mode, N = 512, M = 64:
// 63 -> 27 ms; of 32 vectors, N = 576, M = 64: 19.2 -> 8.5 ms. The backward error
// after one solve of a system of order 2048 is 2.2e-7, 3.0e-7 in FP32 arithmetic.
template <int VT> struct TcSolve {
  static constexpr int KC = 32;                       // columns of a chunk
  static constexpr int AT = SRT * KC, BT = VT * KC;   // elements of a piece
  static constexpr int ABYTES = 6 * AT * 2, BBYTES = 9 * BT * 2;
  static constexpr int IMAGE = 2 * 9 * BT;            // elements of a block solution's image
  static constexpr int SMEM = ABYTES + BBYTES + VT * 8 + 32;
  static constexpr uint32_t TCOLS = 4 * VT;           // leading Re, Im, corrections Re, Im
};
// Element (row, k) of a K-major piece of 32 columns in 8 x 8 core matrices.
__device__ __forceinline__ int piece_off(int r, int k) { return ((r >> 3) * 4 + (k >> 3)) * 64 + (r & 7) * 8 + (k & 7); }

struct TcSolveArgs {
  const cf* LU;
  __nv_bfloat16* xb;  // images of the block solutions: [parity][mode][group][IMAGE]
  cd* x;
  int* err;
  int n, M, nrhs, groups;
};

// Grid (mode, group, tile): the tiles that hold the next block (z = 0) start first.
template <int VT, bool FWD>
__global__ void __launch_bounds__(256, 2) solve_tc_kernel(TcSolveArgs a, int k, int first) {
  using S = TcSolve<VT>;
  extern __shared__ __align__(128) unsigned char sraw[];
  __nv_bfloat16* As = (__nv_bfloat16*)sraw;                // [6 pieces][128 x 32]
  __nv_bfloat16* Xs = (__nv_bfloat16*)(sraw + S::ABYTES);  // [3 pieces][-Im, Re, Im][VT x 32]
  size_t* voff = (size_t*)(sraw + S::ABYTES + S::BBYTES);  // [VT] the vectors in x
  uint64_t* full = (uint64_t*)(voff + VT);                 // chunk of the image has landed
  uint64_t* done = full + 1;                               // products of a chunk are complete
  uint32_t* tbase = (uint32_t*)(done + 1);
  volatile int* fail = (volatile int*)(tbase + 1);
  cf* Bs = (cf*)Xs;                                        // [SB][VT] right-hand side of the next block
  cf* D = (cf*)As;                                         // its triangle, column-major, and
  cf* inv = D + SB * SB;                                   // reciprocals of the diagonal
  const int n = a.n, m = blockIdx.x, g = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int njobs = m == 0 ? a.nrhs : 2 * a.nrhs, job0 = g * VT;
  if (job0 >= njobs) return;
  const int G = min(VT, njobs - job0), nblk = n / SB;
  const cf* L = a.LU + (size_t)m * n * n;
  const int kc = first ? (FWD ? 0 : nblk - 1) : (FWD ? k + 1 : k - 1);  // the next block
  const bool crit = blockIdx.z == 0;
  int r0, rows;
  if (first) { r0 = kc * SB; rows = SB; }
  else if (FWD) { r0 = (k + 1) * SB + SRT * blockIdx.z; rows = min(SRT, n - r0); }
  else { const int e = k * SB - SRT * blockIdx.z; r0 = max(0, e - SRT); rows = e - r0; }
  const int coff = FWD ? 0 : rows - SB;  // the next block's rows within the first tile
  auto image = [&](int kb) { return a.xb + (((size_t)(kb & 1) * (a.M + 1) + m) * a.groups + g) * S::IMAGE; };
  if (tid < VT) {
    int q, ri; bool neg;
    job_of(m, a.M, a.nrhs, job0 + min(tid, G - 1), &q, &ri, &neg);
    voff[tid] = ((size_t)q * a.nrhs + ri) * n;
  }
  if (tid == 0) *fail = 0;
  if (first) {
    __syncthreads();
    for (int e = tid; e < SB * VT; e += 256) {
      const int row = e % SB, v = e / SB;
      Bs[row * VT + v] = v < G ? to_cf(load_x<true>(a.x + voff[v] + r0 + row)) : CF(0.f);
    }
  } else {
    if (warp == 0) tc::tmem_alloc(tbase, S::TCOLS);
    if (tid == 32) {
      tc::mbar_init(full, 1);
      tc::mbar_init(done, 1);
      tc::mbar_fence_init();
    }
    // thread: row tid % 128, columns 16 (tid / 128) .. + 15 of the chunk
    const int ar = tid & 127, ac = (tid >> 7) * 16;
    const cf* F = L + (size_t)(k * SB + ac) * n + r0 + ar;
    cf lv[16];
    auto fetch = [&](int ch) {
#pragma unroll
      for (int c = 0; c < 16; ++c) lv[c] = ar < rows ? F[(size_t)(ch * S::KC + c) * n] : CF(0.f);
    };
    fetch(0);
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    const uint32_t tmem = *tbase;
    auto copy_image = [&](int ch) {
      tc::mbar_expect_tx(full, S::BBYTES);
      tc::bulk_g2s(Xs, image(k) + (size_t)ch * 9 * S::BT, S::BBYTES, full);
    };
    if (tid == 0) copy_image(0);
    bool ok = true;
#pragma unroll
    for (int ch = 0; ch < 2; ++ch) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // 8 columns: one core-matrix row per piece
        __align__(16) __nv_bfloat16 pc[6][8];
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          __nv_bfloat16 pr[3], pi[3];
          split3(lv[8 * h + c].x, pr);
          split3(lv[8 * h + c].y, pi);
#pragma unroll
          for (int q = 0; q < 3; ++q) { pc[q][c] = pr[q]; pc[3 + q][c] = pi[q]; }
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) *(uint4*)(As + q * S::AT + piece_off(ar, ac + 8 * h)) = *(const uint4*)pc[q];
      }
      tc::fence_proxy_async();
      __syncthreads();
      if (tid == 0) {
        if (tc::mbar_wait(full, ch)) {
          constexpr uint32_t id = tc::idesc_bf16_f32(SRT, 2 * VT);
          const uint64_t a0 = tc::desc_noswizzle(tc::smem_u32(As), 128, 512);
          const uint64_t b0 = tc::desc_noswizzle(tc::smem_u32(Xs), 128, 512);
          constexpr uint64_t at = S::AT * 2 / 16, bt = S::BT * 2 / 16;  // 16-byte units
          constexpr int qa[6] = {0, 0, 1, 0, 1, 2}, qb[6] = {0, 1, 0, 2, 1, 0};
#pragma unroll
          for (int ks = 0; ks < S::KC / 16; ++ks)
#pragma unroll
            for (int u = 0; u < 6; ++u) {
              const uint64_t kof = ks * 16, bq = b0 + 3 * qb[u] * bt + kof;  // two core matrices along k
              const uint32_t d = tmem + (u == 0 ? 0 : 2 * VT), acc = ch == 0 && ks == 0 && u <= 1 ? 0u : 1u;
              tc::mma_bf16(d, a0 + qa[u] * at + kof, bq + bt, id, acc);
              tc::mma_bf16(d, a0 + (3 + qa[u]) * at + kof, bq, id, 1u);
            }
        } else {
          *fail = 1;
        }
        tc::commit(done);
      }
      if (ch == 0) {
        fetch(1);
        ok = tc::mbar_wait(done, 0);
        tc::fence_after();
        if (tid == 0) copy_image(1);
      }
    }
    // epilogue: warp w holds rows 32 (w % 4) .. + 31 and half w / 4 of the vectors, 8 at a time
    const int row = 32 * (warp & 3) + lane, vh = (warp >> 2) * (VT / 2);
    const bool in_next = crit && row >= coff && row < coff + SB && row < rows;
    cd xv[8];
    auto fetch_x = [&](int v0) {
#pragma unroll
      for (int v = 0; v < 8; ++v)
        xv[v] = row < rows && v0 + v < G ? load_x<true>(a.x + voff[v0 + v] + r0 + row) : C(0.0);
    };
    fetch_x(vh);
    if (!tc::mbar_wait(done, 1)) ok = false;
    tc::fence_after();
    __syncthreads();  // every warp is past its last use of the operands' space
    if (crit) load_triangle(D, L, n, kc);
#pragma unroll 1
    for (int v0 = vh; v0 < vh + VT / 2; v0 += 8) {
      if (v0 > vh) fetch_x(v0);
      const uint32_t t = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + v0;
      float p[4][8];
      tc::tmem_ld8x4(t, t + VT, t + 2 * VT, t + 3 * VT, p);
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const cd val = xv[v] - wide(CF(p[0][v] + p[2][v], p[1][v] + p[3][v]));
        if (in_next) Bs[(row - coff) * VT + v0 + v] = to_cf(val);
        else if (row < rows && v0 + v < G) store_x<true>(a.x + voff[v0 + v] + r0 + row, val);  // the next block's rows are written solved
      }
    }
    if (!ok) *fail = 1;
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (warp == 0) tc::tmem_dealloc(tmem, S::TCOLS);
    if (*fail) {  // a wait gave up: the host is told; the image's copy lands before the CTA leaves
      if (tid == 0) {
        atomicExch(a.err, 1);
        tc::mbar_wait(full, 1, 1 << 20);
      }
      return;
    }
  }
  if (!crit) return;
  if (first) load_triangle(D, L, n, kc);
  __syncthreads();
  if (!FWD) {
    if (tid < SB) inv[tid] = cone<cf>() / D[tid * SB + tid];
    __syncthreads();
  }
  constexpr int JC = VT / 8;  // vectors of a warp
  const int j0 = warp * JC;
  cf b[2][JC];
  solve_triangle<cf, VT, JC, FWD>(D, inv, Bs, j0, b);
  __nv_bfloat16* xo = image(kc);
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < JC; ++j) {
      const int r = lane + 32 * h, v = j0 + j;
      __nv_bfloat16 pr[3], pi[3];
      split3(b[h][j].x, pr);
      split3(b[h][j].y, pi);
      __nv_bfloat16* xc = xo + (size_t)h * 9 * S::BT + piece_off(v, lane);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        xc[(3 * q) * S::BT] = __hneg(pi[q]);
        xc[(3 * q + 1) * S::BT] = pr[q];
        xc[(3 * q + 2) * S::BT] = pi[q];
      }
      if (v >= G) continue;
      cd val = wide(b[h][j]);
      if (!FWD && job0 + v >= a.nrhs && ((r & 3) == 1 || (r & 3) == 2)) val = -val;  // reflected for -m
      store_x<true>(a.x + voff[v] + kc * SB + r, val);
    }
}

template <int VT, bool FWD> void launch_tc_sweep(const TcSolveArgs& a, cudaStream_t s) {
  const int nblk = a.n / SB, smem = TcSolve<VT>::SMEM;
  smem_optin(solve_tc_kernel<VT, FWD>);
  solve_tc_kernel<VT, FWD><<<dim3(a.M + 1, a.groups, 1), 256, smem, s>>>(a, 0, 1);
  for (int i = 0; i + 1 < nblk; ++i) {
    const int k = FWD ? i : nblk - 1 - i;
    const int rows = FWD ? a.n - (k + 1) * SB : k * SB;
    solve_tc_kernel<VT, FWD><<<dim3(a.M + 1, a.groups, (rows + SRT - 1) / SRT), 256, smem, s>>>(a, k, 0);
  }
}

template <int VT>
void launch_tc_solve(const cf* LU, int n, int M, const int* perm, const cd* rhs, cd* x, int nrhs, void* xb, int* err,
                     cudaStream_t s) {
  TcSolveArgs a{LU, (__nv_bfloat16*)xb, x, err, n, M, nrhs, (2 * nrhs + VT - 1) / VT};
  solve_init_kernel<false><<<dim3((n + 255) / 256, M + 1, std::min(2 * nrhs, 1024)), 256, 0, s>>>(n, M, nrhs, perm,
                                                                                                nullptr, rhs, x);
  launch_tc_sweep<VT, true>(a, s);
  launch_tc_sweep<VT, false>(a, s);
}

template <class TF, int VT, bool FWD, bool PHYS>
void launch_sweep(const SolveArgs<TF>& a, cudaStream_t s) {
  const int nblk = a.n / SB, smem = SolveShape<TF, VT>::SMEM;
  const dim3 g1(1, a.M + 1, a.groups);
  smem_optin(solve_step_kernel<TF, VT, FWD, PHYS>);
  solve_step_kernel<TF, VT, FWD, PHYS><<<g1, 256, smem, s>>>(a, 0, 1);
  for (int i = 0; i + 1 < nblk; ++i) {
    const int k = FWD ? i : nblk - 1 - i;
    const int rows = FWD ? a.n - (k + 1) * SB : k * SB;
    solve_step_kernel<TF, VT, FWD, PHYS><<<dim3((rows + SRT - 1) / SRT, a.M + 1, a.groups), 256, smem, s>>>(a, k, 0);
  }
}

template <class TF, int VT, bool PHYS>
void launch_solve(const TF* LU, int n, int M, const int* perm, const double* sw, const cd* rhs, cd* x, int nrhs,
                  void* xb, cudaStream_t s) {
  SolveArgs<TF> a{LU, (TF*)xb, sw, x, n, M, nrhs, (2 * nrhs + VT - 1) / VT};
  solve_init_kernel<PHYS><<<dim3((n + 255) / 256, M + 1, std::min(2 * nrhs, 1024)), 256, 0, s>>>(n, M, nrhs, perm, sw,
                                                                                               rhs, x);
  launch_sweep<TF, VT, true, PHYS>(a, s);
  launch_sweep<TF, VT, false, PHYS>(a, s);
}

// Vectors per group, complex64: the smallest of 4, 8, 16, 32, 64 that holds a mode's 2 nrhs
// vectors, but 16 up to 1600 and 32 up to 4200 vectors in all modes: a block step waits
// for one warp's part of the triangle, whose chain grows with the vectors of a group, and
// only with many vectors is it bound by the bytes that wider groups save.  Whole solves
// with groups of 16, 32, 64, ms: N = 256: M = 0, 40 sides 2.4, 2.9, 4.2; M = 20, 40 sides
// (1640 vectors) 5.4, 5.7, 7.1; N = 512, M = 20: 40 sides 14.8, 14.6, 16.7; 100 (4100) 32.2,
// 29.1, 29.9.
int cf_group(int M, int nrhs) {
  const long long vectors = (2LL * M + 1) * nrhs;
  const int most = vectors <= 1600 ? 16 : vectors <= 4200 ? 32 : 64;
  const int fit = 2 * nrhs <= 4 ? 4 : 2 * nrhs <= 8 ? 8 : 2 * nrhs <= 16 ? 16 : 2 * nrhs <= 32 ? 32 : 64;
  return std::min(fit, most);
}
int cd_group(int nrhs) { return 2 * nrhs <= 4 ? 4 : 8; }
size_t up256(size_t b) { return (b + 255) & ~(size_t)255; }

}  // namespace

size_t lu_solve_scratch_bytes(int n, int M, int nrhs, bool c64) {
  const int vt = c64 ? cf_group(M, nrhs) : cd_group(nrhs);
  const size_t groups = (2 * (size_t)nrhs + vt - 1) / vt;
  const size_t block = (size_t)SB * vt * (!c64 ? sizeof(cd) : vt <= 8 ? sizeof(cf) : 9 * sizeof(__nv_bfloat16));
  return up256((size_t)(M + 1) * n * 4) + 2 * (size_t)(M + 1) * groups * block;
}

int lu_solve_launches(int n) { return 1 + 2 * (n / SB); }

void lu_solve_prepare(const int* piv, int n, int M, void* scratch, cudaStream_t s) {
  // static and dynamic shared memory together stay below the opt-in limit for any n a body can have
  cudaFuncSetAttribute(perm_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_optin_bytes() - 24 * 1024);
  perm_kernel<<<M + 1, 1024, n * sizeof(int), s>>>(piv, n, (int*)scratch);
}

// Vectors per group, complex128: 4 or 8; more would only lengthen the triangle, the FP64
// pipe being the bound.
void lu_solve_modes(const cd* LU, int n, int M, const double* sw, const cd* rhs, cd* x, int nrhs, void* scratch,
                    cudaStream_t s) {
  const int* perm = (const int*)scratch;
  void* xb = (char*)scratch + up256((size_t)(M + 1) * n * 4);
  if (cd_group(nrhs) == 4) launch_solve<cd, 4, true>(LU, n, M, perm, sw, rhs, x, nrhs, xb, s);
  else launch_solve<cd, 8, true>(LU, n, M, perm, sw, rhs, x, nrhs, xb, s);
}

void lu_correction_solve_c64(const cf* LU, int n, int M, const cd* r, cd* d, int nrhs, void* scratch, int* err,
                             cudaStream_t s) {
  const int* perm = (const int*)scratch;
  void* xb = (char*)scratch + up256((size_t)(M + 1) * n * 4);
  switch (cf_group(M, nrhs)) {
    case 4: launch_solve<cf, 4, false>(LU, n, M, perm, nullptr, r, d, nrhs, xb, s); break;
    case 8: launch_solve<cf, 8, false>(LU, n, M, perm, nullptr, r, d, nrhs, xb, s); break;
    case 16: launch_tc_solve<16>(LU, n, M, perm, r, d, nrhs, xb, err, s); break;
    case 32: launch_tc_solve<32>(LU, n, M, perm, r, d, nrhs, xb, err, s); break;
    default: launch_tc_solve<64>(LU, n, M, perm, r, d, nrhs, xb, err, s); break;
  }
}
