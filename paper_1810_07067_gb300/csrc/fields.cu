// Incident data and far fields (Section 6).
#include <algorithm>
#include "smem.cuh"
#include "fields.cuh"
#include "fields_oz.cuh"

// Fourier coefficients (1/n_theta) sum_t s_t e^{-i m theta_t} of the four ring
// traces smp[n_theta][4] (twiddles tw[t] = e^{-2 pi i t/n_theta}), scaled by
// sE (rows 0, 1) and sH (rows 2, 3).  With n_theta = 2^L q (L <= 4), L
// decimation-in-frequency stages first split each row into 2^L sub-sequences
// of q samples (block bitrev(m mod 2^L) holds the terms of the modes of that
// residue, twiddled), so each mode is a q-term sum instead of n_theta terms;
// then one (mode, row) per thread.  Called by every thread of the CTA;
// smp is overwritten.
__device__ void modal_dft(cd* smp, const cd* tw, int n_theta, int M, int nrhs, int w, int i, int n, cd sE,
                          cd sH, cd* __restrict__ rhs) {
  int L = 0;
  while (L < 4 && ((n_theta >> L) & 1) == 0) ++L;
  for (int st = 0, len = n_theta; st < L; ++st, len >>= 1) {
    const int half = len >> 1, tstep = n_theta / len;
    for (int item = threadIdx.x; item < 4 * (n_theta >> 1); item += blockDim.x) {
      const int a = item & 3, bt = item >> 2;             // row, butterfly
      const int blk = bt / half, t = bt % half;
      const int i0 = blk * len + t, i1 = i0 + half;
      const cd u = smp[4 * i0 + a], v = smp[4 * i1 + a];
      smp[4 * i0 + a] = u + v;
      smp[4 * i1 + a] = (u - v) * tw[t * tstep];
    }
    __syncthreads();
  }
  const int q = n_theta >> L, mask = (1 << L) - 1;
  const double inv = 1.0 / n_theta;
  for (int item = threadIdx.x; item < 4 * (2 * M + 1); item += blockDim.x) {
    const int mq = item >> 2, a = item & 3;
    const int m = mq - M;
    const int mm = ((m % n_theta) + n_theta) % n_theta;
    const int r = mm & mask;
    int blk = 0;
    for (int bit = 0; bit < L; ++bit) blk |= ((r >> bit) & 1) << (L - 1 - bit);
    const int step = (mm >> L) << L;  // twiddle index advance: (mm >> L) 2^L (mod n_theta)
    const cd* x = smp + 4 * blk * q;
    cd acc = C(0.0);
    int idx = 0;
    for (int t = 0; t < q; ++t) {
      acc = fma(x[4 * t + a], tw[idx], acc);
      idx += step;
      if (idx >= n_theta) idx -= n_theta;
    }
    rhs[((size_t)mq * nrhs + w) * n + 4 * i + a] = (a < 2 ? sE : sH) * (inv * acc);
  }
}

// n x v = v_theta t - v_t e_theta at one ring point: (v_theta, -v_t)
__device__ __forceinline__ void traces(const cd v[3], double ct, double st, double rp, double zp, cd* out2) {
  cd vr = ct * v[0] + st * v[1], vth = ct * v[1] - st * v[0];
  out2[0] = vth;
  out2[1] = -(rp * vr + zp * v[2]);
}

// Azimuthal integrals c_m = (1/n) sum_t e^{-i a cos alpha_t} e^{i m alpha_t}, alpha_t = 2 pi t / n,
// of a real argument a (the exterior wavenumber is real): the samples are even
// in alpha and the mirror alpha -> pi - alpha conjugates them, so one real number
// per mode is left,
//   c_m = (1/n) sum_t cos(a cos alpha_t) cos(m alpha_t)      (m even)
//   c_m = (-i/n) sum_t sin(a cos alpha_t) cos(m alpha_t)     (m odd)
// over the quarter t = 0..n/4 (n a multiple of 4; weights 2, 4, .., 4, 2).
// ring_even_coef returns that number, b_m: c_m = b_m or -i b_m by the parity of
// m (b_m or +i b_m for e^{+i a cos alpha}), c_{-m} = c_m.  n/4 sincos and n/4
// multiply-adds per mode replace a complex sum over n samples.

// samples smp[2][R][Q] of one argument a (row row): cos and sin, weighted by 1/n
__device__ __forceinline__ void ring_even_sample(double* smp, int R, int Q, int row, int t, double a, const double* ct,
                                                 int n) {
  double s, c;
  sincos(a * ct[t], &s, &c);
  const double w = (t == 0 || t == Q - 1 ? 2.0 : 4.0) / n;
  smp[row * Q + t] = w * c;
  smp[(R + row) * Q + t] = w * s;
}

__device__ __forceinline__ double ring_even_coef(const double* smp, int R, int Q, int row, int m, const double* ct,
                                                 int n) {
  const double* x = smp + ((m & 1) * R + row) * Q;
  const int step = m % n;
  double acc0 = 0.0, acc1 = 0.0;
  int idx = 0;
  for (int t = 0; t + 1 < Q; t += 2) {
    acc0 = fma(x[t], ct[idx], acc0);
    idx += step;
    if (idx >= n) idx -= n;
    acc1 = fma(x[t + 1], ct[idx], acc1);
    idx += step;
    if (idx >= n) idx -= n;
  }
  if (Q & 1) acc0 = fma(x[Q - 1], ct[idx], acc0);
  return acc0 + acc1;
}

// ---------------------------------------------------------------------------
// Modal data of plane waves.  With d = (d_rho cos phi_d, d_rho sin phi_d, d_z) the
// phase on a node's ring has the coefficients
//   C_m = e^{i k0 z d_z} e^{-i m phi_d} i^m-type c_m(k0 r d_rho)   (ring_even_coef),
// and the traces (V the polarisation of E or H, f the phase, cos and sin shifting m by one)
//   V_theta f          -> i (alpha - beta),
//   -(r' V_r + z' V_z) f -> -(r' (alpha + beta) + z' V_z C_m),
//   alpha = C_{m-1} (V_x - i V_y) / 2,  beta = C_{m+1} (V_x + i V_y) / 2.
// So each (node, wave) needs M + 2 real ring integrals instead of the four
// complex transforms of its sampled traces, and everything that depends on
// the wave alone sits in a table tab[w][q][6]: the factors of b_{m-1}, b_m,
// b_{m+1} for E and for H.
// FP64 pipe: N = 512, M = 64, 96 waves: 1.08 ms (7.91 ms with the four sampled
// traces transformed ring by ring; 0.88 ms with the ring integrals of many waves on
// the tensor cores).

// double-double helpers (error-free transforms) for the wave's rotation e^{-i m phi_d}:
// its phase must not lose digits as m grows
struct dd { double h, l; };
__device__ __forceinline__ dd dd_norm(double h, double l) { const double s = h + l; return dd{s, l - (s - h)}; }
__device__ __forceinline__ dd dd_prod(double a, double b) { const double p = a * b; return dd{p, fma(a, b, -p)}; }
__device__ __forceinline__ dd dd_mul(dd a, dd b) {
  const dd p = dd_prod(a.h, b.h);
  return dd_norm(p.h, p.l + (a.h * b.l + a.l * b.h));
}
__device__ __forceinline__ dd dd_add(dd a, dd b) {
  const double s = a.h + b.h, t = s - a.h;
  return dd_norm(s, ((a.h - (s - t)) + (b.h - t)) + (a.l + b.l));
}
__device__ __forceinline__ dd dd_neg(dd a) { return dd{-a.h, -a.l}; }

__device__ __forceinline__ dd dd_shfl(dd a, int lane) {
  return dd{__shfl_sync(0xffffffffu, a.h, lane), __shfl_sync(0xffffffffu, a.l, lane)};
}
struct ddc { dd x, y; };  // complex
__device__ __forceinline__ ddc ddc_mul(ddc a, ddc b) {
  return ddc{dd_add(dd_mul(a.x, b.x), dd_neg(dd_mul(a.y, b.y))), dd_add(dd_mul(a.x, b.y), dd_mul(a.y, b.x))};
}
__device__ __forceinline__ ddc ddc_shfl(ddc a, int lane) { return ddc{dd_shfl(a.x, lane), dd_shfl(a.y, lane)}; }

// The table of the waves w0..w0 + gridDim.x - 1 (one CTA each), wave[w] =
// (k0 d_rho, k0 d_z), and (first CTA) cost[n_theta] = cos(2 pi t / n_theta).  A chain of
// FP64 operations: warp 0 alone forms the powers of z = e^{-i phi_d}, z^1 .. z^32 by
// doubling (lane l holds z^{l + 1}; five products), then 32 more with each product, while
// the other warps form the cosines (every warp the direction, a binary power per mode:
// M = 16 20.8 us, now 14).
__global__ void __launch_bounds__(128) rhs_wave_kernel(int M, double k0, cd hf, cd sE, cd sH,
                                                       const double* __restrict__ dirs,
                                                       const double* __restrict__ pols, int n_theta,
                                                       cd* __restrict__ tab, double2* __restrict__ wave,
                                                       double* __restrict__ cost) {
  extern __shared__ __align__(16) char smem[];
  cd* em = (cd*)smem;  // [M + 2] e^{-i m phi_d}
  const int w = blockIdx.x;
  const double* d = dirs + 3 * w;
  const double* e = pols + 3 * w;
  if (threadIdx.x >= 32) {
    if (w == 0)
      for (int t = threadIdx.x - 32; t < n_theta; t += 96) cost[t] = cospi(2.0 * t / n_theta);
  } else {
    const int lane = threadIdx.x;
    const dd s2 = dd_add(dd_prod(d[0], d[0]), dd_prod(d[1], d[1]));
    ddc z{dd{1.0, 0.0}, dd{0.0, 0.0}};
    double drho = 0.0;
    if (s2.h > 1e-280) {
      const double r0 = rsqrt(s2.h);
      const dd t = dd_mul(s2, dd_prod(r0, r0));
      const dd r = dd_norm(r0, 0.5 * r0 * ((1.0 - t.h) - t.l));
      z.x = dd_mul(dd{d[0], 0.0}, r);
      z.y = dd_neg(dd_mul(dd{d[1], 0.0}, r));
      drho = s2.h * r.h + (s2.h * r.l + s2.l * r.h);
    }
    if (lane == 0) {
      wave[w] = make_double2(k0 * drho, k0 * d[2]);
      em[0] = C(1.0);
    }
    ddc p = z;
#pragma unroll
    for (int n = 1; n < 32; n <<= 1) {  // lanes 0..n - 1 hold z^1 .. z^n
      const ddc q = ddc_mul(ddc_shfl(p, n - 1), ddc_shfl(p, lane & (n - 1)));
      if (lane >= n) p = q;
    }
    const ddc z32 = ddc_shfl(p, 31);
    for (int m0 = 1; m0 < M + 2; m0 += 32) {
      if (m0 > 1) p = ddc_mul(p, z32);
      if (m0 + lane < M + 2) em[m0 + lane] = C(p.x.h, p.y.h);
    }
  }
  __syncthreads();
  const double hv[3] = {d[1] * e[2] - d[2] * e[1], d[2] * e[0] - d[0] * e[2], d[0] * e[1] - d[1] * e[0]};
  auto cm = [&](int m) {  // e^{-i m phi_d} times the unit of c_m
    const int a = abs(m);
    cd v = em[a];
    if (m < 0) v = conj(v);
    return (a & 1) ? mul_i(v) : v;
  };
  for (int it = threadIdx.x; it < 2 * (2 * M + 1); it += blockDim.x) {
    const int q = it >> 1, h = it & 1, m = q - M;
    const double* V = h ? hv : e;
    const cd sc = h ? sH * hf : sE;
    cd* o = tab + ((size_t)w * (2 * M + 1) + q) * 6 + 3 * h;
    o[0] = sc * (cm(m - 1) * C(0.5 * V[0], -0.5 * V[1]));
    o[1] = sc * (V[2] * cm(m));
    o[2] = sc * (cm(m + 1) * C(0.5 * V[0], 0.5 * V[1]));
  }
}

// One CTA per (R nodes, wave): samples of the nodes' ring phases, their
// coefficients b_m, then two rows (E or H) per (mode, node) and thread.  An SM's FP64 pipe
// issues a warp's operation in 19 clocks, so a call that leaves SMs without a CTA takes
// fewer nodes a CTA: N = 128, M = 16, one wave, 8 nodes 11 us, 2 nodes 7 us.
template <int R>
__global__ void __launch_bounds__(256) rhs_kernel(FieldGeom g, int M, const double2* __restrict__ wave,
                                                  const cd* __restrict__ tab, const double* __restrict__ cost,
                                                  int w0, int nrhs, int n, cd* __restrict__ rhs) {
  extern __shared__ __align__(16) char smem[];
  const int Q = n / 4 + 1;
  double* ct = (double*)smem;           // [n], n a multiple of 4
  double* smp = ct + n;                 // [2][R][Q]
  double* b = smp + 2 * R * Q;      // [M + 2][R]
  double2* phz = (double2*)(b + R * (M + 2));  // [R] e^{i k0 z d_z}
  const int i0 = blockIdx.x * R, w = blockIdx.y;
  const double2 wv = wave[w];
  for (int t = threadIdx.x; t < n; t += blockDim.x) ct[t] = cost[t];
  if (threadIdx.x < R) {
    double s, c;
    sincos(wv.y * g.z[i0 + threadIdx.x], &s, &c);
    phz[threadIdx.x] = make_double2(c, s);
  }
  __syncthreads();
  for (int it = threadIdx.x; it < R * Q; it += blockDim.x) {
    const int row = it / Q, t = it - row * Q;
    ring_even_sample(smp, R, Q, row, t, wv.x * g.r[i0 + row], ct, n);
  }
  __syncthreads();
  for (int it = threadIdx.x; it < R * (M + 2); it += blockDim.x)
    b[it] = ring_even_coef(smp, R, Q, it % R, it / R, ct, n);
  __syncthreads();
  const cd* tw = tab + (size_t)w * (2 * M + 1) * 6;
  for (int it = threadIdx.x; it < 2 * R * (2 * M + 1); it += blockDim.x) {
    const int h = it & 1, row = (it >> 1) % R, q = (it >> 1) / R, m = q - M, i = i0 + row;
    const cd* u = tw + (size_t)q * 6 + 3 * h;
    const cd al = b[abs(m - 1) * R + row] * u[0], be = b[abs(m + 1) * R + row] * u[2];
    const cd D = b[abs(m) * R + row] * u[1];
    cd* o = rhs + ((size_t)q * nrhs + w0 + w) * (4 * g.N) + 4 * i + 2 * h;
    const cd pz = C(phz[row].x, phz[row].y);
    o[0] = mul_i(al - be) * pz;
    o[1] = -((g.rp[i] * (al + be) + g.zp[i] * D) * pz);
  }
}

// Sampled incident fields EH[w][i][t][6] (E then H, Cartesian) at the ring
// points of node i -> modal data, as rhs_kernel.
__global__ void rhs_samples_kernel(FieldGeom g, int M, cd sE, cd sH, const cd* __restrict__ EH, int nrhs,
                                   int n_theta, cd* __restrict__ rhs) {
  extern __shared__ __align__(16) char smem[];
  cd* smp = (cd*)smem;
  cd* tw = smp + 4 * n_theta;
  const int i = blockIdx.x, w = blockIdx.y;
  const double rp = g.rp[i], zp = g.zp[i];
  const cd* src = EH + ((size_t)w * g.N + i) * n_theta * 6;
  for (int t = threadIdx.x; t < n_theta; t += blockDim.x) {
    double ct, st;
    sincospi(2.0 * t / n_theta, &st, &ct);
    tw[t] = C(ct, -st);
    traces(src + 6 * t, ct, st, rp, zp, smp + 4 * t);
    traces(src + 6 * t + 3, ct, st, rp, zp, smp + 4 * t + 2);
  }
  __syncthreads();
  modal_dft(smp, tw, n_theta, M, nrhs, w, i, 4 * g.N, sE, sH, rhs);
}

void launch_rhs_samples(const FieldGeom& g, int M, cd sE, cd sH, const cd* EH, int nrhs, int n_theta, cd* rhs,
                        cudaStream_t s) {
  int smem = n_theta * 5 * (int)sizeof(cd);
  smem_optin(rhs_samples_kernel);
  rhs_samples_kernel<<<dim3(g.N, nrhs), 256, smem, s>>>(g, M, sE, sH, EH, nrhs, n_theta, rhs);
}

size_t rhs_planewave_scratch_doubles(int M, int nrhs, int n_theta) {
  const size_t nw = nrhs < RHS_WAVES ? nrhs : RHS_WAVES;
  return nw * ((size_t)(2 * M + 1) * 12 + 2) + n_theta;
}

// N is a multiple of 16.  Waves pass RHS_WAVES at a time, so the table stays
// below 1 KiB x (2M + 1) x 96 bytes whatever the number of waves.
// Ring integrals of fewer multiply-adds than this stay on the FP64 pipe with the rest
// of the data (two launches instead of five): N = 512, M = 64: 8 waves (1.3e7) 0.17 ms
// there and 0.20 ms on the tensor cores, 32 waves (5e7) 0.43 and 0.40 ms, 96 waves
// (1.6e8) 1.08 and 0.88 ms; N = 128, M = 16, 200 waves (1e7) 0.29 and 0.31 ms.
#define RHS_FMA_MIN 4e7
size_t rhs_planewave_work_bytes(int N, int M, int nrhs, int n_theta) {
  const double fma = (double)N * nrhs * (M + 2.0) * (n_theta / 4);
  return fma >= RHS_FMA_MIN ? rhs_plan(N, M, n_theta, nrhs, pass_bytes()).bytes : 0;
}

bool launch_rhs_planewave(const FieldGeom& g, int M, double k0, double omega, cd mu0, cd sE, cd sH,
                          const double* dirs_dev, const double* pols_dev, int nrhs, int n_theta, double* scratch,
                          void* work, size_t work_bytes, cd* rhs, int* err, cudaStream_t s) {
  RhsPlan plan{};
  if (work) {
    plan = rhs_plan(g.N, M, n_theta, nrhs, pass_bytes());
    if (plan.bytes > work_bytes) return false;
  }
  const int Q = n_theta / 4 + 1;
  const int smem_w = (M + 2) * (int)sizeof(cd);
  if (smem_w > 48 * 1024) smem_optin(rhs_wave_kernel);
  const int nw = nrhs < RHS_WAVES ? nrhs : RHS_WAVES;
  const int R = (long long)(g.N / 8) * nw < 152 ? 2 : 8;  // nodes of a CTA: N is a multiple of 16
  const int smem = (n_theta + 2 * R * Q + R * (M + 4)) * (int)sizeof(double);
  if (smem > 48 * 1024) R == 2 ? smem_optin(rhs_kernel<2>) : smem_optin(rhs_kernel<8>);
  cd* tab = (cd*)scratch;
  double2* wave = (double2*)(tab + (size_t)nw * (2 * M + 1) * 6);
  double* cost = (double*)(wave + nw);
  const cd hf = C(k0) / (omega * mu0);  // H polarisation (k0 / (omega mu0)) d x e
  for (int w0 = 0; w0 < nrhs; w0 += RHS_WAVES) {
    const int c = nrhs - w0 < RHS_WAVES ? nrhs - w0 : RHS_WAVES;
    const cd one = C(1.0);  // the tensor-core form applies the traces' factors itself
    rhs_wave_kernel<<<c, 128, smem_w, s>>>(M, k0, work ? one : hf, work ? one : sE, work ? one : sH,
                                           dirs_dev + 3 * (size_t)w0, pols_dev + 3 * (size_t)w0, n_theta, tab, wave, cost);
    if (work) launch_rhs_products(g, M, wave, tab, sE, sH * hf, w0, c, nrhs, n_theta, plan, work, rhs, err, s);
    else if (R == 2) rhs_kernel<2><<<dim3(g.N / 2, c), 256, smem, s>>>(g, M, wave, tab, cost, w0, nrhs, n_theta, rhs);
    else rhs_kernel<8><<<dim3(g.N / 8, c), 256, smem, s>>>(g, M, wave, tab, cost, w0, nrhs, n_theta, rhs);
  }
  return true;
}

// Currents on the node rings: cur[w][i][t][a] = sum_m x[m][w][4i+a] e^{i m theta_t}
// (CART false: the four components on (t, e_theta); true: J and M in Cartesian
// components, six values, and pts[i][t] = the ring point and its surface weight).
// Modes +-m are joined (x_m + x_-m with the cosine, i (x_m - x_-m) with the
// sine), and so are the azimuths t and n - t (even and odd part): 4 multiply-adds
// per component, mode pair and azimuth pair, the cosines from one table.
// Vectors w0 .. w0 + gridDim.y - 1 of the nrhs.
template <bool CART>
__global__ void __launch_bounds__(128) ring_kernel(FieldGeom g, int M, const cd* __restrict__ x, int w0, int nrhs,
                                                   int n_theta, cd* __restrict__ cur, double4* __restrict__ pts) {
  extern __shared__ __align__(16) char smem[];
  cd* Sm = (cd*)smem;          // [M + 1][4]
  cd* Dm = Sm + 4 * (M + 1);   // [M + 1][4]
  cd* tw = Dm + 4 * (M + 1);   // [n_theta]
  const int i = blockIdx.x, w = blockIdx.y;
  const int n = 4 * g.N;
  for (int it = threadIdx.x; it < 4 * (M + 1); it += blockDim.x) {
    const int m = it >> 2, a = it & 3;
    const cd u = x[((size_t)(M + m) * nrhs + w0 + w) * n + 4 * i + a];
    const cd v = x[((size_t)(M - m) * nrhs + w0 + w) * n + 4 * i + a];
    Sm[it] = m ? u + v : u;
    Dm[it] = mul_i(u - v);
  }
  for (int t = threadIdx.x; t < n_theta; t += blockDim.x) {
    double s, c;
    sincospi(2.0 * t / n_theta, &s, &c);
    tw[t] = C(c, s);
  }
  __syncthreads();
  const double rp = g.rp[i], zp = g.zp[i];
  for (int t = threadIdx.x; t <= n_theta / 2; t += blockDim.x) {
    cd a[4] = {C(0.0), C(0.0), C(0.0), C(0.0)}, b[4] = {C(0.0), C(0.0), C(0.0), C(0.0)};
    int idx = 0;
    for (int m = 0; m <= M; ++m) {
      const cd e = tw[idx];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        a[u] = fma(e.x, Sm[4 * m + u], a[u]);
        b[u] = fma(e.y, Dm[4 * m + u], b[u]);
      }
      idx += t;
      if (idx >= n_theta) idx -= n_theta;
    }
    for (int mir = 0; mir < 2; ++mir) {
      const int tm = mir ? n_theta - t : t;
      if (mir && (t == 0 || tm == t)) break;
      cd v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = mir ? a[u] - b[u] : a[u] + b[u];
      if (!CART) {
        cd* dst = cur + (((size_t)w * g.N + i) * n_theta + tm) * 4;
#pragma unroll
        for (int u = 0; u < 4; ++u) dst[u] = v[u];
      } else {
        const double c = tw[tm].x, s = tw[tm].y;
        cd* dst = cur + (((size_t)w * g.N + i) * n_theta + tm) * 6;
#pragma unroll
        for (int h = 0; h < 2; ++h) {  // t = r' e_r + z' e_z, e_theta = (-s, c, 0)
          dst[3 * h] = (rp * c) * v[2 * h] - s * v[2 * h + 1];
          dst[3 * h + 1] = (rp * s) * v[2 * h] + c * v[2 * h + 1];
          dst[3 * h + 2] = zp * v[2 * h];
        }
        if (w == 0) {
          const double r = g.r[i];
          pts[(size_t)i * n_theta + tm] = make_double4(r * c, r * s, g.z[i], g.w[i] * r * (6.283185307179586 / n_theta));
        }
      }
    }
  }
}

template <bool CART>
static void launch_ring(const FieldGeom& g, int M, const cd* x, int w0, int wc, int nrhs, int n_theta, cd* cur,
                        double4* pts, cudaStream_t s) {
  smem_optin(ring_kernel<CART>);
  ring_kernel<CART><<<dim3(g.N, wc), 128, (8 * (M + 1) + n_theta) * sizeof(cd), s>>>(g, M, x, w0, nrhs, n_theta, cur,
                                                                                  pts);
}

// One CTA per (rhs, direction): Jh, Mh by the ring quadrature, then E_oo.
__global__ void farfield_kernel(FieldGeom g, cd k0, double omega, cd eps0, const cd* __restrict__ cur, int nrhs,
                                const double* __restrict__ dirs, int ndir, int n_theta, cd* __restrict__ E) {
  const int dix = blockIdx.x, w = blockIdx.y;
  const double xh0 = dirs[3 * dix], xh1 = dirs[3 * dix + 1], xh2 = dirs[3 * dix + 2];
  cd J[3] = {C(0.0), C(0.0), C(0.0)}, Mv[3] = {C(0.0), C(0.0), C(0.0)};
  const long long total = (long long)g.N * n_theta;
  const double TWO_PI = 6.283185307179586;
  for (long long it = threadIdx.x; it < total; it += blockDim.x) {
    int i = (int)(it / n_theta), t = (int)(it % n_theta);
    double s, c;
    sincospi(2.0 * t / n_theta, &s, &c);
    double r = g.r[i], z = g.z[i];
    double proj = xh0 * r * c + xh1 * r * s + xh2 * z;
    double da = g.w[i] * r * (TWO_PI / n_theta);
    cd ph = da * cexpi(-(k0 * proj));
    const cd* cv = cur + (((size_t)w * g.N + i) * n_theta + t) * 4;
    // t = r' e_r + z' e_z ; e_theta = (-s, c, 0)
    double tx = g.rp[i] * c, ty = g.rp[i] * s, tz = g.zp[i];
    cd j1 = ph * cv[0], j2 = ph * cv[1], m1 = ph * cv[2], m2 = ph * cv[3];
    J[0] += tx * j1 - s * j2; J[1] += ty * j1 + c * j2; J[2] += tz * j1;
    Mv[0] += tx * m1 - s * m2; Mv[1] += ty * m1 + c * m2; Mv[2] += tz * m1;
  }
  __shared__ cd red[6][32];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  cd vals[6] = {J[0], J[1], J[2], Mv[0], Mv[1], Mv[2]};
#pragma unroll
  for (int a = 0; a < 6; ++a) {
    for (int o = 16; o > 0; o >>= 1) {
      vals[a].x += __shfl_xor_sync(0xffffffffu, vals[a].x, o);
      vals[a].y += __shfl_xor_sync(0xffffffffu, vals[a].y, o);
    }
    if (lane == 0) red[a][wid] = vals[a];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    cd tot[6];
    for (int a = 0; a < 6; ++a) {
      tot[a] = C(0.0);
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) tot[a] += red[a][q];
    }
    cd xJ = xh0 * tot[0] + xh1 * tot[1] + xh2 * tot[2];
    cd pre = -(k0 * k0) / (C(0.0, omega) * eps0);
    double xh[3] = {xh0, xh1, xh2};
    cd cr[3];
    cr[0] = xh1 * tot[5] - xh2 * tot[4];
    cr[1] = xh2 * tot[3] - xh0 * tot[5];
    cr[2] = xh0 * tot[4] - xh1 * tot[3];
    cd ik = mul_i(k0);
    double inv4pi = 1.0 / (4.0 * 3.141592653589793);
    cd* dst = E + ((size_t)w * ndir + dix) * 3;
    for (int a = 0; a < 3; ++a) dst[a] = inv4pi * (pre * (tot[a] - xh[a] * xJ) + ik * cr[a]);
  }
}

void launch_far_field(const FieldGeom& g, int M, cd k0, double omega, cd eps0, const cd* x, int nrhs,
                      const double* dirs_dev, int ndir, int n_theta, cd* cur, cd* E, cudaStream_t s) {
  launch_ring<false>(g, M, x, 0, nrhs, nrhs, n_theta, cur, nullptr, s);
  farfield_kernel<<<dim3(ndir, nrhs), 256, 0, s>>>(g, k0, omega, eps0, cur, nrhs, dirs_dev, ndir, n_theta, E);
}

// ---------------------------------------------------------------------------
// Fields at points off the surface: E = cJ curl curl S J + cM curl S M,
// H = dM curl curl S M + dJ curl S J (eqs. exteriorfield, interiorfield,
// interior_dual with the region's constants), with
//   curl S V      = sum G (ik - 1/R) Rh x V da,
//   curl curl S V = sum G [(k^2 + ik/R - 1/R^2) V + (-k^2 - 3ik/R + 3/R^2)(Rh.V) Rh] da
// over the node rings (ds-weights x trapezoid in theta).  One CTA per (point,
// split of the ring points, WR right-hand sides): the kernels of a (point,
// ring point) pair are formed once for WR right-hand sides, ring points and
// Cartesian currents come from ring_kernel, and the partial sums of the splits
// are joined by nearfield_join_kernel.  FP64 pipe; N = 320, M = 32, 2 sides, 100
// points: 2.7 ms with the rings (8.4 ms with one CTA per point and side, which
// left a second wave on a third of the SMs and formed the kernels per side; 1.6 ms on
// the tensor cores, which take all but few pairs).
template <int WR>
__global__ void __launch_bounds__(128) nearfield_kernel(long long total, const double4* __restrict__ pts,
                                                        const cd* __restrict__ cur, const double* __restrict__ X,
                                                        int nrhs, cd k, long long per, cd* __restrict__ part) {
  const int p = blockIdx.x, sp = blockIdx.y, w0 = blockIdx.z * WR;
  const double x0 = X[3 * p], x1 = X[3 * p + 1], x2 = X[3 * p + 2];
  cd acc[WR][12];  // curl curl S J, curl S M, curl curl S M, curl S J (3 components each)
#pragma unroll
  for (int v = 0; v < WR; ++v)
#pragma unroll
    for (int a = 0; a < 12; ++a) acc[v][a] = C(0.0);
  const cd ik = mul_i(k), k2 = k * k;
  const double FOUR_PI = 12.566370614359172;
  const long long it1 = min(total, (sp + 1) * per);
  for (long long it = sp * per + threadIdx.x; it < it1; it += blockDim.x) {
    const double4 y = pts[it];
    const double R0 = x0 - y.x, R1 = x1 - y.y, R2 = x2 - y.z;
    const double R = sqrt(R0 * R0 + R1 * R1 + R2 * R2), iR = 1.0 / R;
    const double hv[3] = {R0 * iR, R1 * iR, R2 * iR};
    double sn, cs;
    sincos(k.x * R, &sn, &cs);
    double am = y.w * iR / FOUR_PI;
    if (k.y != 0.0) am *= exp(-(k.y * R));
    const cd G = C(am * cs, am * sn);
    const cd c1 = G * (ik - C(iR));
    const cd aa = G * (k2 + iR * ik - C(iR * iR));
    const cd bb = G * (C(3.0 * iR * iR) - k2 - (3.0 * iR) * ik);
#pragma unroll
    for (int v = 0; v < WR; ++v) {
      if (WR > 1 && w0 + v >= nrhs) break;
      const cd* cv = cur + ((size_t)(w0 + v) * total + it) * 6;
#pragma unroll
      for (int h = 0; h < 2; ++h) {  // J, then M
        const cd V0 = cv[3 * h], V1 = cv[3 * h + 1], V2 = cv[3 * h + 2];
        const cd bp = bb * (hv[0] * V0 + hv[1] * V1 + hv[2] * V2);
        cd* cc = acc[v] + 6 * h;
        cc[0] = fma(hv[0], bp, fma(aa, V0, cc[0]));
        cc[1] = fma(hv[1], bp, fma(aa, V1, cc[1]));
        cc[2] = fma(hv[2], bp, fma(aa, V2, cc[2]));
        const cd W0 = c1 * V0, W1 = c1 * V1, W2 = c1 * V2;
        cd* cu = acc[v] + (h ? 3 : 9);
        cu[0] = fma(hv[1], W2, fma(-hv[2], W1, cu[0]));
        cu[1] = fma(hv[2], W0, fma(-hv[0], W2, cu[1]));
        cu[2] = fma(hv[0], W1, fma(-hv[1], W0, cu[2]));
      }
    }
  }
  __shared__ cd red[12][4];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int v = 0; v < WR; ++v) {
#pragma unroll
    for (int a = 0; a < 12; ++a) {
      for (int o = 16; o > 0; o >>= 1) {
        acc[v][a].x += __shfl_xor_sync(0xffffffffu, acc[v][a].x, o);
        acc[v][a].y += __shfl_xor_sync(0xffffffffu, acc[v][a].y, o);
      }
      if (lane == 0) red[a][wid] = acc[v][a];
    }
    __syncthreads();
    if (threadIdx.x < 12 && w0 + v < nrhs)
      part[(((size_t)(w0 + v) * gridDim.x + p) * gridDim.y + sp) * 12 + threadIdx.x] =
          (red[threadIdx.x][0] + red[threadIdx.x][1]) + (red[threadIdx.x][2] + red[threadIdx.x][3]);
    __syncthreads();
  }
}

// out[w][p][6] from the splits' partial sums: one thread per (point, component)
__global__ void nearfield_join_kernel(long long items, int splits, const cd* __restrict__ part, cd cJ, cd cM, cd dM,
                                      cd dJ, cd* __restrict__ out) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= items) return;
  const long long wp = t / 6;
  const int c = (int)(t - 6 * wp), d = c % 3, a0 = c < 3 ? d : 6 + d;
  const cd* src = part + wp * splits * 12;
  cd u = C(0.0), v = C(0.0);
  for (int q = 0; q < splits; ++q) { u += src[12 * q + a0]; v += src[12 * q + a0 + 3]; }
  out[t] = c < 3 ? cJ * u + cM * v : dM * u + dJ * v;
}

// Splits of the ring points: enough CTAs for four per SM, each thread at least
// eight ring points (the sums across the CTA cost about as much as two).
static int near_field_splits(long long total, int nt, int nrhs) {
  const long long ctas = (long long)nt * ((nrhs + 1) / 2);
  const long long want = (608 + ctas - 1) / ctas, most = std::max(1LL, total / (128 * 8));
  return (int)std::max(1LL, std::min({want, most, 1024LL}));
}

// Right-hand sides per pass: their ring currents stay within 8 GB (or are one).
int near_field_group(long long total, int nrhs) {
  return (int)std::max(1LL, std::min<long long>(nrhs, 8000000000LL / (96 * total)));
}

size_t near_field_part(long long total, int nt, int nrhs) {
  const int group = near_field_group(total, nrhs), last = nrhs % group ? nrhs % group : group;
  return (size_t)nt * 12 * std::max(group * near_field_splits(total, nt, group), last * near_field_splits(total, nt, last));
}

// Fewer (point, ring point) pairs than NF_PAIRS_MIN stay on the FP64 pipe, whose kernel
// needs no digits: N = 128, M = 16, 10 points, one side (1.5e5) 0.17 ms there and 0.23 ms
// on the tensor cores, 50 points (8e5) 0.41 and 0.39 ms; N = 320, M = 32, 100 points (5e6)
// one side 1.83 and 1.55 ms, two 2.74 and 1.56 ms, eight 10.6 and 2.5 ms.
// So do points that fill too little of their row tiles of 128 (18 rows a point), whose
// digits are copied and multiplied whole, for the sides that share the tiles:
// nf_fills_rows.  N = 576, M = 64, targets 0.02 from the surface (2.8e6 ring points), one
// side: one point 2.7 ms there and 4.2 ms on the tensor cores, four 4.2 and 5.1, seven 6.7
// and 5.9, eight (two tiles) 6.3 and 7.1, thirty 21 and 18; two sides, one 4.6 and 6.2,
// four 6.9 and 7.0; eight sides, one 16.7 and 20.3, two 20.0 and 20.6, four 27 and 21.
#define NF_PAIRS_MIN 7e5
static bool nf_fills_rows(int nt, int nrhs) {
  const double row_tiles = (double)tiles((size_t)NF_ROWS * nt, OZ_RT);
  return nt * (20.0 + 7.0 * nrhs) >= OZ_RT * row_tiles;
}
size_t near_field_work_bytes(long long total, int nt, int nrhs) {
  const int group = near_field_group(total, nrhs);
  return (double)total * nt >= NF_PAIRS_MIN && nf_fills_rows(nt, group) ? nf_plan(total, nt, group, pass_bytes()).bytes : 0;
}

bool launch_near_field(const FieldGeom& g, int M, const cd* x, int nrhs, const double* X_dev, int nt, int n_theta,
                       cd k, cd cJ, cd cM, cd dM, cd dJ, cd* cur, double* pts, cd* part, void* work, size_t work_bytes,
                       cd* out, int* err, cudaStream_t s) {
  const long long total = (long long)g.N * n_theta;
  const int group = near_field_group(total, nrhs);
  NfPlan plan{};
  if (work) {
    plan = nf_plan(total, nt, group, pass_bytes());
    if (plan.bytes > work_bytes) return false;
  }
  for (int w0 = 0; w0 < nrhs; w0 += group) {
    const int wc = std::min(group, nrhs - w0), splits = near_field_splits(total, nt, wc);
    const long long per = (total + splits - 1) / splits;
    launch_ring<true>(g, M, x, w0, wc, nrhs, n_theta, cur, (double4*)pts, s);
    if (work) {
      launch_nearfield_products(total, (const double4*)pts, cur, X_dev, nt, wc, k, cJ, cM, dM, dJ, plan, work,
                                out + (size_t)w0 * nt * 6, err, s);
      continue;
    }
    if (wc == 1)
      nearfield_kernel<1><<<dim3(nt, splits, 1), 128, 0, s>>>(total, (const double4*)pts, cur, X_dev, wc, k, per, part);
    else
      nearfield_kernel<2><<<dim3(nt, splits, (wc + 1) / 2), 128, 0, s>>>(total, (const double4*)pts, cur, X_dev, wc, k,
                                                                         per, part);
    const long long items = (long long)wc * nt * 6;
    nearfield_join_kernel<<<(unsigned)((items + 127) / 128), 128, 0, s>>>(items, splits, part, cJ, cM, dM, dJ,
                                                                          out + (size_t)w0 * nt * 6);
  }
  return true;
}

// ---------------------------------------------------------------------------
// Far field on a (polar x azimuth) grid, mode by mode.  For x_hat at polar
// angle theta and azimuth phi, substituting theta' = phi + alpha on each ring
// turns eq. farfieldform into E(theta, phi) = R_z(phi) sum_m e^{i m phi} F_m(theta),
// with F_m the far-field vector of mode m in the frame (e_rho, e_phi, e_z) of
// azimuth phi, where x_hat = (sin theta, 0, cos theta).  The ring integrals
// need c_m = (1/n) sum_t e^{-i a cos alpha_t} e^{i m alpha_t}, a = k0 r sin theta
// (same trapezoid rule in alpha as mueller_far_field):
//   (1/2pi) int e^{-i a cos} e^{i m alpha} {1, cos, sin} = {c_m, (c_{m+1}+c_{m-1})/2, (c_{m+1}-c_{m-1})/(2i)}.
// c_m = b_m (m even) or -i b_m (m odd), the real b_m from ring_even_coef.

// coef[m][p][j] = b_m(k0 r_j sin theta_p), m = 0..M + 1, and phase[p][j] = 2 pi w_j r_j
// e^{-i k0 z_j cos theta_p}, for the P2 = ceil(n_polar / 2) upper polar angles
// (theta_{n-1-p} = pi - theta_p has the same b and the conjugate phase).  One
// CTA per (polar angle, FFC_R nodes).  FP64 pipe: per (p, j) n/4 sincos and
// (M + 2) n/4 multiply-adds.
#define FFC_R 8
__global__ void __launch_bounds__(256) ffgrid_coef_kernel(FieldGeom g, int M, double k0, int n_polar, int n,
                                                          double* __restrict__ coef, double2* __restrict__ phase) {
  extern __shared__ __align__(16) char smem[];
  const int Q = n / 4 + 1, P2 = gridDim.x;
  double* ct = (double*)smem;      // [n] cos(2 pi t / n)
  double* smp = ct + n;            // [2][FFC_R][Q]
  const int p = blockIdx.x, j0 = blockIdx.y * FFC_R;
  double sth, cth;
  sincospi((p + 0.5) / n_polar, &sth, &cth);
  for (int t = threadIdx.x; t < n; t += blockDim.x) ct[t] = cospi(2.0 * t / n);
  __syncthreads();
  for (int it = threadIdx.x; it < FFC_R * Q; it += blockDim.x) {
    const int row = it / Q, t = it - row * Q;
    if (j0 + row < g.N) ring_even_sample(smp, FFC_R, Q, row, t, g.r[j0 + row] * sth * k0, ct, n);
  }
  if (threadIdx.x < FFC_R && j0 + threadIdx.x < g.N) {
    const int j = j0 + threadIdx.x;
    double s, c;
    sincos(k0 * (g.z[j] * cth), &s, &c);
    const double wr = 6.283185307179586 * g.w[j] * g.r[j];
    phase[(size_t)p * g.N + j] = make_double2(wr * c, -wr * s);
  }
  __syncthreads();
  for (int it = threadIdx.x; it < FFC_R * (M + 2); it += blockDim.x) {
    const int row = it % FFC_R, m = it / FFC_R, j = j0 + row;
    if (j < g.N) coef[((size_t)m * P2 + p) * g.N + j] = ring_even_coef(smp, FFC_R, Q, row, m, ct, n);
  }
}

// F[w][p][q][3] for mode m = q - M, polar angles p and n_polar - 1 - p.  With
// U_a the sums over the nodes of phase c_{m+a} X_a for X_{+-1} = r' J1 +- i J2 and
// X_0 = z' J1 (and the same of M), J_rho = (U_+ + U_-)/2, J_phi = (U_+ - U_-)/(2i),
// J_z = U_0; the real and imaginary parts of the phase are summed apart (A, B),
// so the two mirrored angles are A + iB and A - iB: 4 multiply-adds per term
// for both.  FP64 pipe: 24 multiply-adds per node, mode, angle pair and side; the
// whole grid, N = 512, M = 64, 8 sides, 180 x 360: 3.93 ms (49.2 ms with complex
// coefficients per angle and the phase formed per mode and side; 0.81 ms on the
// tensor cores, which take all but small grids).  One CTA per
// (mode, PT polar angles, WT right-hand sides); a thread owns one (angle, side)
// and every JS-th node; the nodes pass through shared memory JC at a time.
// PT is 16, and 2 for at most four angles, whose 16-angle tiles would be idle lanes that
// the FP64 pipe issues all the same: N = 128, M = 16, 8 sides, one direction 126 -> 24 us.
template <int PT, int WT>
__global__ void __launch_bounds__(128) ffgrid_mode_kernel(FieldGeom g, int M, double k0, double omega, cd eps0,
                                                          int n_polar, int P2, const double* __restrict__ coef,
                                                          const double2* __restrict__ phase,
                                                          const cd* __restrict__ x, int nrhs, cd* __restrict__ F) {
  constexpr int JS = 128 / (PT * WT), JC = JS > 16 ? JS : 16;
  __shared__ double2 sb[3][JC][PT + 1];  // b_{m+1}, b_m, b_{m-1} times the phase's (cos, sin)
  __shared__ cd sX[JC][WT][6];
  __shared__ cd red[PT == 16 ? (JS > 1 ? 128 : 1) : 12 * 4 * PT * WT];
  const int q = blockIdx.y, m = q - M, p0 = blockIdx.x * PT, w0 = blockIdx.z * WT;
  const int tid = threadIdx.x, pl = tid % PT, wl = (tid / PT) % WT, js = tid / (PT * WT);
  const int n = 4 * g.N;
  const int mi[3] = {abs(m + 1), abs(m), abs(m - 1)};
  cd A[6], B[6];
#pragma unroll
  for (int u = 0; u < 6; ++u) { A[u] = C(0.0); B[u] = C(0.0); }
  for (int j0 = 0; j0 < g.N; j0 += JC) {  // N is a multiple of 16
    const int nj = JC == 16 ? JC : min(JC, g.N - j0);
    for (int it = tid; it < JC * PT; it += 128) {
      const int jj = it % JC, pp = it / JC;
      if (p0 + pp < P2 && jj < nj) {
        const size_t o = (size_t)(p0 + pp) * g.N + j0 + jj;
        const double2 ph = phase[o];
#pragma unroll
        for (int u = 0; u < 3; ++u) {
          const double b = coef[(size_t)mi[u] * P2 * g.N + o];
          sb[u][jj][pp] = make_double2(b * ph.x, b * ph.y);
        }
      }
    }
    for (int it = tid; it < JC * WT * 2; it += 128) {
      const int h = it & 1, jj = (it >> 1) % JC, w = (it >> 1) / JC, j = j0 + jj;
      if (jj >= nj) continue;
      cd v1 = C(0.0), v2 = C(0.0);
      if (w0 + w < nrhs) {
        const cd* xv = x + ((size_t)q * nrhs + w0 + w) * n + 4 * j + 2 * h;
        v1 = xv[0];
        v2 = mul_i(xv[1]);
      }
      const cd r1 = g.rp[j] * v1;
      sX[jj][w][3 * h] = r1 + v2;
      sX[jj][w][3 * h + 1] = g.zp[j] * v1;
      sX[jj][w][3 * h + 2] = r1 - v2;
    }
    __syncthreads();
    if (p0 + pl < P2) {
#pragma unroll 2
      for (int jj = js; jj < nj; jj += JS) {
#pragma unroll
        for (int u = 0; u < 6; ++u) {
          const double2 b = sb[u % 3][jj][pl];
          const cd X = sX[jj][wl][u];
          A[u] = fma(b.x, X, A[u]);
          B[u] = fma(b.y, X, B[u]);
        }
      }
    }
    __syncthreads();
  }
  if constexpr (PT < 16) {  // the nodes' parts of a warp, then of the four warps
    constexpr int L = PT * WT;
    const int lane = tid & 31, wid = tid >> 5;
#pragma unroll
    for (int v = 0; v < 12; ++v) {
      cd t = v < 6 ? A[v % 6] : B[v % 6];
#pragma unroll
      for (int o = L; o < 32; o <<= 1) {
        t.x += __shfl_xor_sync(0xffffffffu, t.x, o);
        t.y += __shfl_xor_sync(0xffffffffu, t.y, o);
      }
      if (lane < L) red[(v * 4 + wid) * L + lane] = t;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < 12; ++v) {
      const cd* x4 = red + v * 4 * L + lane % L;
      const cd t = (x4[0] + x4[L]) + (x4[2 * L] + x4[3 * L]);
      if (v < 6) A[v % 6] = t;
      else B[v % 6] = t;
    }
  } else if (JS > 1) {
    for (int v = 0; v < 12; ++v) {
      red[tid] = v < 6 ? A[v % 6] : B[v % 6];
      __syncthreads();
      cd t = C(0.0);
#pragma unroll
      for (int k = 0; k < JS; ++k) t += red[k * PT * WT + tid % (PT * WT)];
#pragma unroll
      for (int u = 0; u < 6; ++u) {
        if (v == u) A[u] = t;
        if (v == 6 + u) B[u] = t;
      }
      __syncthreads();
    }
  }
  const int p = p0 + pl, w = w0 + wl;
  if (js != 0 || p >= P2 || w >= nrhs) return;
  ffgrid_vector(A, B, m, M, k0, omega, eps0, p, n_polar, F + (size_t)w * n_polar * (2 * M + 1) * 3);
}

// E[w][p][s][3] (Cartesian) = R_z(phi_s) sum_m e^{i m phi_s} F_m: one CTA per
// (polar angle, rhs).  Modes +-m are joined (F_m + F_-m with the cosine,
// i (F_m - F_-m) with the sine) and so are the azimuths s and n - s (even and
// odd part): 4 multiply-adds per component, mode pair and azimuth pair.
__global__ void __launch_bounds__(128) ffgrid_synth_kernel(int M, int n_polar, int n_azim, const cd* __restrict__ F,
                                                           int nrhs, cd* __restrict__ E) {
  extern __shared__ __align__(16) char smem[];
  const int nq = 2 * M + 1;
  cd* Sm = (cd*)smem;          // [M + 1][3] F_m + F_-m (F_0 for m = 0)
  cd* Dm = Sm + 3 * (M + 1);   // [M + 1][3] i (F_m - F_-m)
  cd* tw = Dm + 3 * (M + 1);   // [n_azim] e^{2 pi i s / n_azim}
  const int p = blockIdx.x, w = blockIdx.y;
  const cd* src = F + ((size_t)w * n_polar + p) * nq * 3;
  for (int t = threadIdx.x; t < 3 * (M + 1); t += blockDim.x) {
    const int m = t / 3, a = t - 3 * m;
    const cd u = src[(M + m) * 3 + a], v = src[(M - m) * 3 + a];
    Sm[t] = m ? u + v : u;
    Dm[t] = mul_i(u - v);
  }
  for (int s = threadIdx.x; s < n_azim; s += blockDim.x) {
    double sn, cs;
    sincospi(2.0 * s / n_azim, &sn, &cs);
    tw[s] = C(cs, sn);
  }
  __syncthreads();
  for (int s = threadIdx.x; s <= n_azim / 2; s += blockDim.x) {
    cd a[3] = {C(0.0), C(0.0), C(0.0)}, b[3] = {C(0.0), C(0.0), C(0.0)};
    int idx = 0;
    for (int m = 0; m <= M; ++m) {
      const cd e = tw[idx];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        a[u] = fma(e.x, Sm[3 * m + u], a[u]);
        b[u] = fma(e.y, Dm[3 * m + u], b[u]);
      }
      idx += s;
      if (idx >= n_azim) idx -= n_azim;
    }
    for (int mir = 0; mir < 2; ++mir) {
      const int sm = mir ? n_azim - s : s;
      if (mir && (s == 0 || sm == s)) break;
      const cd cphi = tw[sm];  // (cos phi, sin phi)
      const cd v0 = mir ? a[0] - b[0] : a[0] + b[0], v1 = mir ? a[1] - b[1] : a[1] + b[1];
      cd* dst = E + (((size_t)w * n_polar + p) * n_azim + sm) * 3;
      dst[0] = cphi.x * v0 - cphi.y * v1;
      dst[1] = cphi.y * v0 + cphi.x * v1;
      dst[2] = mir ? a[2] - b[2] : a[2] + b[2];
    }
  }
}

template <int PT, int WT>
static void launch_ffgrid_mode(const FieldGeom& g, int M, double k0, double omega, cd eps0, int n_polar, int P2,
                               const double* coef, const double2* phase, const cd* x, int nrhs, cd* F,
                               cudaStream_t s) {
  ffgrid_mode_kernel<PT, WT><<<dim3((P2 + PT - 1) / PT, 2 * M + 1, (nrhs + WT - 1) / WT), 128, 0, s>>>(
      g, M, k0, omega, eps0, n_polar, P2, coef, phase, x, nrhs, F);
}

// Sums of fewer multiply-adds than this stay on the FP64 pipe (three launches; the
// tensor-core form takes a dozen and cuts every operand into digits): N = 128, M = 32,
// 60 angles, one side (6e6) 0.14 ms there and 0.18 ms on the tensor cores; N = 256,
// M = 64, 90 angles, one side (4e7) 0.37 and 0.29 ms; M = 32, eight sides 0.60 and
// 0.31 ms; N = 512, M = 64, 180 angles, one side (1.4e8) 1.17 and 0.55 ms, eight sides
// 3.34 and 0.86 ms.
#define FFO_MIN 2e7
size_t far_field_grid_work_bytes(int N, int M, int n_polar, int n_azim, int n_alpha, int nrhs) {
  const double fma = 24.0 * ((n_polar + 1) / 2) * N * (2.0 * M + 1.0) * nrhs;
  return fma >= FFO_MIN ? ffo_plan(N, M, n_polar, n_azim, n_alpha, nrhs, pass_bytes()).bytes : 0;
}

size_t far_field_grid_coef_doubles(int N, int M, int n_polar) {
  return (size_t)((n_polar + 1) / 2) * N * (M + 4);  // M + 2 coefficients and the complex phase
}

bool launch_far_field_grid(const FieldGeom& g, int M, double k0, double omega, cd eps0, const cd* x, int nrhs,
                           int n_polar, int n_azim, int n_alpha, double* coef, void* work, size_t work_bytes, cd* F, cd* E,
                           int* err, cudaStream_t s) {
  if (work) {
    const FfoPlan plan = ffo_plan(g.N, M, n_polar, n_azim, n_alpha, nrhs, pass_bytes());
    if (plan.bytes > work_bytes) return false;
    launch_ffgrid_products(g, M, k0, omega, eps0, x, nrhs, n_polar, n_azim, n_alpha, plan, work, F, E, err, s);
    return true;
  }
  const int P2 = (n_polar + 1) / 2, Q = n_alpha / 4 + 1;
  double2* phase = (double2*)coef;                 // 16-byte aligned at the block's start
  double* b = coef + 2 * (size_t)P2 * g.N;
  const int smem1 = (n_alpha + 2 * FFC_R * Q) * (int)sizeof(double);
  smem_optin(ffgrid_coef_kernel);
  ffgrid_coef_kernel<<<dim3(P2, (g.N + FFC_R - 1) / FFC_R), 256, smem1, s>>>(g, M, k0, n_polar, n_alpha, b, phase);
  // right-hand sides per CTA: the smallest of 1, 2, 4, 8 that holds them (the
  // angles' coefficients are read once per group); with few angles fewer, as long as
  // there are SMs for the CTAs (one direction, 8 sides a CTA, 4, 2, 1: N = 128, M = 16,
  // 8 sides 38, 26, 21, 24 us; N = 512, M = 64, 4 sides 110, 65, 58, 78 us)
  int wt = nrhs <= 1 ? 1 : nrhs <= 2 ? 2 : nrhs <= 4 ? 4 : 8;
  if (P2 <= 4) {
    while (wt > 1 && (long long)((P2 + 1) / 2) * (2 * M + 1) * ((nrhs + wt - 1) / wt) < 152) wt /= 2;
    if (wt == 1) launch_ffgrid_mode<2, 1>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
    else if (wt == 2) launch_ffgrid_mode<2, 2>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
    else if (wt == 4) launch_ffgrid_mode<2, 4>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
    else launch_ffgrid_mode<2, 8>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
  } else if (wt == 1) launch_ffgrid_mode<16, 1>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
  else if (wt == 2) launch_ffgrid_mode<16, 2>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
  else if (wt == 4) launch_ffgrid_mode<16, 4>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
  else launch_ffgrid_mode<16, 8>(g, M, k0, omega, eps0, n_polar, P2, b, phase, x, nrhs, F, s);
  const int smem3 = (6 * (M + 1) + n_azim) * (int)sizeof(cd);
  smem_optin(ffgrid_synth_kernel);
  ffgrid_synth_kernel<<<dim3(n_polar, nrhs), 128, smem3, s>>>(M, n_polar, n_azim, F, nrhs, E);
  return true;
}

// Currents at refined nodes: xs[v][4s + a] = sum_k Lm[s][k] x[v][4 (node0[s] + k) + a]
// (v over modes x right-hand sides; the 16 nodes of sub-node s's panel);
// grid.y strides over the vectors.
__global__ void interp_currents_kernel(const cd* __restrict__ x, int n, int nsub, const int* __restrict__ node0,
                                       const double* __restrict__ Lm, long long nvec, cd* __restrict__ xs) {
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 4 * nsub) return;
  const int s = idx >> 2, a = idx & 3;
  const double* L = Lm + (size_t)s * 16;
  for (long long v = blockIdx.y; v < nvec; v += gridDim.y) {
    const cd* xv = x + v * n + 4 * node0[s] + a;
    cd acc = C(0.0);
#pragma unroll
    for (int k = 0; k < 16; ++k) acc = fma(L[k], xv[4 * k], acc);
    xs[v * 4 * nsub + idx] = acc;
  }
}

void launch_interp_currents(const cd* x, int n, int nsub, const int* node0, const double* Lm, long long nvec, cd* xs,
                            cudaStream_t s) {
  const unsigned gy = (unsigned)(nvec < 65535 ? nvec : 65535);
  interp_currents_kernel<<<dim3((4 * nsub + 255) / 256, gy), 256, 0, s>>>(x, n, nsub, node0, Lm, nvec, xs);
}
