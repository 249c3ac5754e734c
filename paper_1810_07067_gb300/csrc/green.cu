// Modal Green's functions, their target derivatives and the per-mode Mueller
// blocks, on the GPU.
//
// For a target (r_t, z_t) and a source (r_s, z_s) the nine spectra
//   F0 = g^{k0}_m, F1 = g^{k1}_m                                 (eq. green11)
//   F2, F3 = d/dr_t, d/dz_t of g^{k0}_m; F4, F5 the same for k1    (eq. firstder)
//   F6, F7, F8 = d2/dr_t2, d2/dr_t dz_t, d2/dz_t2 of (g^{k0} - g^{k1})_m
//                                                       (Section 4.3, differences)
// are computed for m = 0..M+1 from nphi azimuthal samples of the integrand
// and a cosine transform (the integrands are even in phi).  Where the half
// grid fits one exact digit product (nphi/2 + 1 <= 272 samples) the transform
// runs on the tensor cores: support pairs in chunks (support_sample_kernel,
// oz_real_gemm_kernel, support_post_kernel), far pairs binned by their own
// grid (far_sample_kernel, oz_real_gemm_kernel, far_assemble_kernel);
// otherwise each pair's warp sums it directly (far_kernel, support_kernel).
//
// Kernel splitting (Section 4): with u = rho^2 and G = exp(ik sqrt u)/(4pi sqrt u),
// every family is written as  a(phi) u^{-1/2} + beta u^{-3/2} + c(phi)  with
// a, c entire in phi and beta a per-pair constant (the r_t - r_s cos(phi)
// factors are rewritten as alpha_r + u/(2 r_t) so that only a constant
// multiplies u^{-3/2}).  The u^{-1/2} part is the discrete convolution of eq.
// discA, computed as the transform of a(phi_j) times the band-limited samples
// of u^{-1/2} (the "D^{-1}(f . D q)" form); the u^{-3/2} part is beta times the
// closed-form coefficient of eq. pm.  The Fourier coefficients of u^{-1/2} and
// u^{-3/2} are (2 r_t r_s)^{-1/2} P_m(chi) and (2 r_t r_s)^{-3/2} S_m(chi) with
// P_m = sqrt(8) Q_{m-1/2} (eq. lm, recurrence eq. recurform, Miller's backward
// recurrence when the forward one is unstable) and S_m from the appendix
// relation.  Splitting is used only when the plain trapezoid rule would alias
// above the requested accuracy (zeta^{nphi-M-1} > eps, zeta = chi - sqrt(chi^2-1)).
#include <cuda_runtime.h>
#include <cstdio>
#include "smem.cuh"
#include "green.cuh"
#include "block.cuh"
#include "grid.cuh"
#include "digits.cuh"
#include "ozaki.cuh"

__constant__ SeriesTables c_tab;

void upload_series_tables(const SeriesTables& t) { cudaMemcpyToSymbol(c_tab, &t, sizeof(SeriesTables)); }

// ---------------------------------------------------------------------------
// Laplace-type modal coefficients, one thread per split pair.
// pairs: [n][4] = (r_t, z_t, r_t - r_s, z_t - z_s); leg: [(Mq+1)+Ms][n] index-major:
// rows 0..Mq hold P^_n = P_n / sqrt(B), rows Mq+1.. hold S^_m = S_m / B^{3/2}.
// rinv[k] = 1 / (2k + 1) for k < nr (shared memory): the recurrences divide by
// odd integers at every step.
//
// With c = chi - 1 and E_m = 2 D_m = 2 (P_{m-1} - P_m) the recurrence (2m+1) P_{m+1} = 4 m
// chi P_m - (2m-1) P_{m-1} keeps the O(1) differences accurate when chi -> 1:
//   up:   P_m = P_{m-1} - E_m / 2,  E_{m+1} = w - (w + E_m) / (2m + 1), w = E_m - 4 c P_m
//   down: P_m = P_{m+1} + E_{m+1} / 2,  E_m = w + (w + E_{m+1}) / (2m - 1), w = E_{m+1} + 4 c P_m
// four FP64 operations a step, on one serial chain per pair: the kernel is bound
// by that chain when the pairs are few and by the FP64 pipe when they are many.
// Downward (Miller) the start is arbitrary and its error, like every rounding on
// the way, falls by zeta^2 a step: the steps from m* = M_q + 19.6 / l (l =
// ln(1/zeta)) to M_q + 11.5 / l run in FP32, whose rounding of 6e-8 is below
// 1e-17 at M_q; then FP64 to mode 0 for the normalisation P_0, and once more from
// M_q with the normalised values, stored as they come. (One FP64 pass from m* with
// a division a step and unscaled values rescaled in memory took 250 us for the
// 64-node sphere; modal_kernels of 64 pairs as a whole fell from 311 to 157 us and
// the sphere from 4.29 to 4.11 ms with this form.)
__host__ __device__ void legendre_one(double rt, double dr, double dz, long long p, long long n, int Mq, int Ms,
                                      double* __restrict__ leg, const double* rinv, int nr) {
  auto inv_odd = [&](int k) { return k < nr ? rinv[k] : 1.0 / (2.0 * k + 1.0); };  // 1 / (2k + 1)
  const double rs = rt - dr;
  const double d2 = dr * dr + dz * dz, B = 2.0 * rt * rs;
  const double c = d2 / B, cp1 = 2.0 + c, c4 = 4.0 * c;  // chi - 1, chi + 1
  double K, E;
  ellipke(sqrt(c / cp1), &K, &E);
  const double scp1 = sqrt(cp1), isB = 1.0 / sqrt(B), isB3 = isB * isB * isB;
  const double P0 = 4.0 * K / scp1;
  const double lz = log1p(c + sqrt(c) * scp1);  // -ln(zeta)
  double* Pv = leg;                                // rows 0..Mq: P^_m
  double* Sv = leg + (long long)(Mq + 1) * n;      // rows 0..Ms-1: S^_m
  // S_m = (1 - 2m)(chi P_m - P_{m-1})/(chi^2 - 1) = (2m - 1)(D_m - c P_m)/(c (c + 2)), of P^ = P isB
  const double sfac = 0.5 * isB * isB / (c * cp1), c2 = 2.0 * c;
  Sv[p] = 4.0 * E / (c * scp1) * isB3;
  const double LN32 = 3.4657359027997265;
  if (2.0 * Mq * lz <= LN32) {
    double P = P0 * isB, e = 2.0 * (4.0 * scp1 * E - c * P0) * isB;  // P^_0, E_1
    double k = 1.0;                                                 // 2m - 1
    Pv[p] = P;
    for (int m = 1; m <= Mq; ++m) {
      P = fma(-0.5, e, P);
      Pv[(long long)m * n + p] = P;
      if (m < Ms) {
        Sv[(long long)m * n + p] = k * sfac * fma(-c2, P, e);
        k += 2.0;
      }
      const double w = fma(-c4, P, e);
      e = fma(-inv_odd(m), w + e, w);
    }
  } else {
    // P~_{m*+1} = 0, E~_{m*+1} = 2, down to M_q
    const int mstar = Mq + (int)ceil(19.6 / lz) + 2, m32 = Mq + (int)ceil(11.5 / lz) + 2;
    float Pf = 0.f, ef = 2.f;
    const float c4f = (float)c4;
    for (int m = mstar; m > m32; --m) {
      Pf = fmaf(0.5f, ef, Pf);
      const float w = fmaf(c4f, Pf, ef);
      ef = fmaf((float)inv_odd(m - 1), w + ef, w);
    }
    double P = (double)Pf, e = (double)ef;
    int m = mstar > m32 ? m32 : mstar;
    for (; m > Mq; --m) {
      P = fma(0.5, e, P);
      const double w = fma(c4, P, e);
      e = fma(inv_odd(m - 1), w + e, w);
    }
    const double Pq = P, eq = e;  // P_{Mq+1}, E_{Mq+1}
    for (; m >= 1; --m) {
      P = fma(0.5, e, P);
      const double w = fma(c4, P, e);
      e = fma(inv_odd(m - 1), w + e, w);
    }
    const double scale = P0 * isB / fma(0.5, e, P);  // P_0
    P = Pq * scale;
    e = eq * scale;
    double k = 2.0 * Ms - 3.0;  // 2m - 1
    for (m = Mq; m >= 0; --m) {
      P = fma(0.5, e, P);
      Pv[(long long)m * n + p] = P;
      const double w = fma(c4, P, e);
      e = m >= 1 ? fma(inv_odd(m - 1), w + e, w) : 0.0;
      if (m >= 1 && m < Ms) {
        Sv[(long long)m * n + p] = k * sfac * fma(-c2, P, e);
        k -= 2.0;
      }
    }
  }
}

// Entries of the reciprocal table: the largest index either recurrence reaches
// (the Miller start Mq + ceil(19.6 / ln(1/zeta)) + 2 with ln(1/zeta) above
// ln(32) / (2 Mq) on that branch), capped at 96 KiB of shared memory.
static int legendre_table_entries(int Mq) {
  const long long need = (long long)Mq + (long long)(19.6 * 2.0 * Mq / 3.4657359027997265) + 4;
  return (int)std::min<long long>(need, 96 * 1024 / 8);
}

__device__ __forceinline__ void fill_odd_reciprocals(double* rinv, int nr) {
  for (int k = threadIdx.x; k < nr; k += blockDim.x) rinv[k] = 1.0 / (2.0 * k + 1.0);
  __syncthreads();
}

__global__ void legendre_kernel(const double* __restrict__ pairs, long long n, int Mq, int Ms,
                                double* __restrict__ leg, int nr) {
  extern __shared__ double rinv[];
  fill_odd_reciprocals(rinv, nr);
  long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= n) return;
  legendre_one(pairs[4 * p], pairs[4 * p + 2], pairs[4 * p + 3], p, n, Mq, Ms, leg, rinv, nr);
}

void launch_legendre(const double* pairs, long long n, int Mq, int Ms, double* leg, cudaStream_t s) {
  if (n <= 0) return;
  const int tpb = 128, nr = legendre_table_entries(Mq);
  smem_optin(legendre_kernel);
  legendre_kernel<<<(unsigned)((n + tpb - 1) / tpb), tpb, nr * 8, s>>>(pairs, n, Mq, Ms, leg, nr);
}

// ---------------------------------------------------------------------------
// One warp computes the nine spectra of one pair into shared memory.
// Shared layout per warp: smp[NFAM*H] (cd), spec[NFAM*Ms] (cd), q[H] (double),
// phs[Mq+1] (double).
int green_smem_per_warp(const GreenParams& gp) { return green_smem_bytes(gp); }

struct WarpSmem {
  cd* smp; cd* spec; double* q; double* phs;
};

__device__ __forceinline__ WarpSmem warp_smem(const GreenParams& gp, char* base) {
  WarpSmem w;
  w.smp = (cd*)base;
  w.spec = w.smp + NFAM * gp.H;
  w.q = (double*)(w.spec + NFAM * gp.Ms);
  w.phs = w.q + gp.H;
  return w;
}


// ---------------------------------------------------------------------------
// One sample of the nine kernels (times 4 pi) at u = rho^2 = d2 + 4 r_t r_s s2,
// s2 = sin^2(phi / 2): out[f * stride], weighted by w.
//
// With the functions of special.cuh (sample_*), per wavenumber
//   E = c / rho + i k sinc,  E' = (k^2 a / 2) / rho - 1 / (2 rho^3) + i k^3 sig1 / 2,
// the difference of E'' is (k0^4 eta0 - k1^4 eta1) / rho - g0 / (2 rho^3) + i (k0^5 sig2_0
// - k1^5 sig2_1) / 4, g0 = -(k0^2 - k1^2) / 4, and a split pair has its band-limited
// samples q in the place of 1 / rho with the rho^-3 parts rewritten (see the top
// of the file).  Where both |k| rho >= 2 a pair that is not split takes E, E' and
// E'' from exp(i k rho) directly; the difference does not cancel there.
// K0R, K1R: real wavenumbers in real arithmetic.  FP64 pipe: about 180
// operations a sample for two real wavenumbers (600 with the seven entire functions
// of each wavenumber and complex products by zero parts): far pairs of the N = 1024,
// M = 128 body 64 -> 21 ms, its support pairs 26 -> 16.5 ms, the lossy cylinder's
// (N = 576, M = 64) 36 -> 16 and 13.6 -> 7.4 ms.
struct PairSample {
  double d2, rr4, dr0, rs2, zd;  // rr4 = 4 r_t r_s, rs2 = 2 r_s
  double irt, alpha;             // split pairs
};

// k^p of a real or complex wavenumber
template <bool R> __device__ __forceinline__ auto kval(const cd& z) {
  if constexpr (R) return z.x;
  else return z;
}
// a + i b for real or complex a, b
__device__ __forceinline__ cd join(double a, double b) { return C(a, b); }
__device__ __forceinline__ cd join(cd a, cd b) { return C(a.x - b.y, a.y + b.x); }
__device__ __forceinline__ double fun_fma2(double s, double x, double c) { return fma(s, x, c); }
__device__ __forceinline__ cd fun_fma2(double s, cd x, cd c) { return fma(s, x, c); }
__device__ __forceinline__ double dif(double a, double b) { return a - b; }
__device__ __forceinline__ cd dif(double a, cd b) { return C(a - b.x, -b.y); }
__device__ __forceinline__ cd dif(cd a, cd b) { return a - b; }

template <bool R>
__device__ __forceinline__ auto sample_fun(const KPow& kp, double su, double u, double isu) {
  if constexpr (R) {
    const double x = kp.k.x * su;
    if (kp.ak * su < 2.0) return sample_series<double>(c_tab, x * x);
    double s, c;
    sincos(x, &s, &c);
    const double xi = kp.ik.x * isu;
    return sample_closed<double>(s, c, xi, xi * xi);
  } else {
    const cd x = su * kp.k;
    if (kp.ak * su < 2.0) return sample_series<cd>(c_tab, u * kp.k2);
    cd s, c;
    csincos(x, &s, &c);
    const cd xi = isu * kp.ik;
    return sample_closed<cd>(s, c, xi, xi * xi);
  }
}

// E, E', E'' (times w) from exp(i k rho); isw = w / rho
template <bool R>
__device__ __forceinline__ void sample_direct(const KPow& kp, double su, double iu, double isw, cd* E) {
  const double a1 = 0.5 * iu * isw, a2 = 0.5 * iu * a1;
  if constexpr (R) {
    const double x = kp.k.x * su;
    double s, c;
    sincos(x, &s, &c);
    const double p = fma(-x, x, 3.0), x3 = 3.0 * x;
    E[0] = C(c * isw, s * isw);
    E[1] = C(a1 * fma(-x, s, -c), a1 * fma(x, c, -s));
    E[2] = C(a2 * fma(p, c, x3 * s), a2 * fma(p, s, -(x3 * c)));
  } else {
    const cd ikr = mul_i(su * kp.k), e = cexpi(su * kp.k);
    E[0] = isw * e;
    E[1] = a1 * (e * (ikr - C(1.0)));
    E[2] = a2 * (e * (ikr * ikr - 3.0 * ikr + C(3.0)));
  }
}

template <bool K0R, bool K1R>
__device__ __forceinline__ void pair_sample(const GreenParams& gp, const PairSample& ps, double s2, double w, bool split,
                                            double q, cd* __restrict__ out, int stride) {
  const double u = fma(ps.rr4, s2, ps.d2);
  const double isu = rsqrt(u);
  double su = u * isu;
  su = fma(0.5 * isu, fma(-su, su, u), su);  // sqrt(u)
  const double rd2 = 2.0 * fma(ps.rs2, s2, ps.dr0), zd2 = 2.0 * ps.zd;
  if (!split && fmin(gp.kp0.ak, gp.kp1.ak) * su >= 2.0) {
    const double iu = isu * isu;
    cd E0[3], E1[3];
    sample_direct<K0R>(gp.kp0, su, iu, w * isu, E0);
    sample_direct<K1R>(gp.kp1, su, iu, w * isu, E1);
    out[0] = E0[0]; out[stride] = E1[0];
    out[2 * stride] = rd2 * E0[1]; out[3 * stride] = zd2 * E0[1];
    out[4 * stride] = rd2 * E1[1]; out[5 * stride] = zd2 * E1[1];
    const cd D1 = E0[1] - E1[1], D2 = E0[2] - E1[2], t1 = D1 + D1;
    out[6 * stride] = fma(rd2 * rd2, D2, t1);
    out[7 * stride] = (rd2 * zd2) * D2;
    out[8 * stride] = fma(zd2 * zd2, D2, t1);
    return;
  }
  const auto f0 = sample_fun<K0R>(gp.kp0, su, u, isu);
  const auto f1 = sample_fun<K1R>(gp.kp1, su, u, isu);
  // real-part and imaginary-part functions (complex for a complex wavenumber)
  const auto G0 = (0.5 * kval<K0R>(gp.kp0.k2)) * f0.a;
  const auto G1 = (0.5 * kval<K1R>(gp.kp1.k2)) * f1.a;
  const auto P0 = (0.5 * kval<K0R>(gp.kp0.k3)) * f0.sig1;
  const auto P1 = (0.5 * kval<K1R>(gp.kp1.k3)) * f1.sig1;
  const auto eta = dif(kval<K0R>(gp.kp0.k4) * f0.eta, kval<K1R>(gp.kp1.k4) * f1.eta);
  const auto dPP = dif((0.25 * kval<K0R>(gp.kp0.k5)) * f0.sig2, (0.25 * kval<K1R>(gp.kp1.k5)) * f1.sig2);
  const auto dG = dif(G0, G1), dP = dif(P0, P1);
  const auto g0 = kval<K0R && K1R>(gp.gamma0);
  const double v = w * (split ? q : isu);  // weight of the 1 / rho parts
  out[0] = join(v * f0.c, w * (kval<K0R>(gp.kp0.k) * f0.sinc));
  out[stride] = join(v * f1.c, w * (kval<K1R>(gp.kp1.k) * f1.sinc));
  const double wr = w * rd2, wz = w * zd2, vr = v * rd2, vz = v * zd2;
  const auto i2 = dP + dP;
  if (!split) {
    const double h = 0.5 * isu * isu;  // E' = (G - h) / rho + i P
    out[2 * stride] = join(vr * fun_add(G0, -h), wr * P0); out[3 * stride] = join(vz * fun_add(G0, -h), wz * P0);
    out[4 * stride] = join(vr * fun_add(G1, -h), wr * P1); out[5 * stride] = join(vz * fun_add(G1, -h), wz * P1);
    const auto d2r = eta - h * g0, r2 = dG + dG;
    out[6 * stride] = join(v * fun_fma2(rd2 * rd2, d2r, r2), w * fun_fma2(rd2 * rd2, dPP, i2));
    out[7 * stride] = join((vr * zd2) * d2r, (wr * zd2) * dPP);
    out[8 * stride] = join(v * fun_fma2(zd2 * zd2, d2r, r2), w * fun_fma2(zd2 * zd2, dPP, i2));
  } else {
    const double h = 0.5 * ps.irt;
    out[2 * stride] = join(v * fun_add(rd2 * G0, -h), wr * P0); out[3 * stride] = join(vz * G0, wz * P0);
    out[4 * stride] = join(v * fun_add(rd2 * G1, -h), wr * P1); out[5 * stride] = join(vz * G1, wz * P1);
    const auto r2 = dG + dG;
    const double rda = fma(0.5, rd2, ps.alpha) * ps.irt, zr = ps.zd * ps.irt;
    out[6 * stride] = join(v * (fun_fma2(rd2 * rd2, eta, r2) - rda * g0), w * fun_fma2(rd2 * rd2, dPP, i2));
    out[7 * stride] = join(v * ((rd2 * zd2) * eta - zr * g0), (wr * zd2) * dPP);
    out[8 * stride] = join(v * fun_fma2(zd2 * zd2, eta, r2), w * fun_fma2(zd2 * zd2, dPP, i2));
  }
}

// The weighted samples W.smp[f][j] = w_j F_f(phi_j), j = 0..nl/2 (w = 1/2 at
// both ends), of one pair on its grid g: the first half of warp_pair_spectra,
// by the threads t = 0..NT-1 of a group whose barrier is sync().
// RR: real wavenumbers, 2 both, 1 k0 only, 0 neither, -1 decided at run time.
template <int NT, int RR = -1, class Sync>
__device__ __forceinline__ void group_pair_samples(const GreenParams& gp, double rt, double dr0, double zd,
                                                   long long sid, const double* __restrict__ leg, long long n_split,
                                                   const double* __restrict__ cosT, const WarpSmem& W, int t,
                                                   const PairGrid& g, const Sync& sync) {
  const int Mq = gp.Mq, mask = gp.nphi - 1;
  const int nl = g.nl;  // local grid size; sample j sits at entry j of its tables
  const double* __restrict__ s2L = g.s2L;
  const int H = nl / 2 + 1, Q = nl / 4;  // samples on [0, pi]; fold point
  const double rs = rt - dr0;
  const double d2 = dr0 * dr0 + zd * zd;
  const double alpha = dr0 - d2 / (2.0 * rt);
  const bool split = sid >= 0;
  const double TWO_PI = 6.283185307179586;
  if (split) {  // dec == 1
    for (int nn = t; nn <= Mq; nn += NT) W.phs[nn] = leg[(long long)nn * n_split + sid];
    sync();
    // q_j = (P^_0 + 2 sum_n P^_n cos(n phi_j)) / 2pi, folded: even n give E, odd n give O,
    // q_j = E + O and q_{n/2 - j} = E - O
    for (int j = t; j <= Q; j += NT) {
      double e = 0.0, o = 0.0;
      for (int nn = 1; nn <= Mq; nn += 2) o = fma(W.phs[nn], cosT[(nn * j) & mask], o);
      for (int nn = 2; nn <= Mq; nn += 2) e = fma(W.phs[nn], cosT[(nn * j) & mask], e);
      e = W.phs[0] + 2.0 * e;
      o = 2.0 * o;
      W.q[j] = (e + o) / TWO_PI;
      W.q[H - 1 - j] = (e - o) / TWO_PI;
    }
    sync();
  }
  PairSample ps;
  ps.d2 = d2; ps.rr4 = 4.0 * rt * rs; ps.dr0 = dr0; ps.rs2 = 2.0 * rs; ps.zd = zd;
  ps.irt = 1.0 / rt; ps.alpha = alpha;
  for (int j = t; j < H; j += NT) {
    const double wj = (j == 0 || j == H - 1) ? 0.5 : 1.0;
    cd* out = W.smp + j;
    if (RR == 2 || (RR < 0 && gp.k0_real && gp.k1_real))
      pair_sample<true, true>(gp, ps, s2L[j], wj, split, split ? W.q[j] : 0.0, out, H);
    else if (RR == 1 || (RR < 0 && gp.k0_real))
      pair_sample<true, false>(gp, ps, s2L[j], wj, split, split ? W.q[j] : 0.0, out, H);
    else if (RR <= 0)
      pair_sample<false, false>(gp, ps, s2L[j], wj, split, split ? W.q[j] : 0.0, out, H);
  }
  sync();
}

__device__ void warp_pair_samples(const GreenParams& gp, double rt, double dr0, double zd,
                                  long long sid, const double* __restrict__ leg, long long n_split,
                                  const double* __restrict__ cosT, const WarpSmem& W, int lane,
                                  const PairGrid& g) {
  group_pair_samples<32>(gp, rt, dr0, zd, sid, leg, n_split, cosT, W, lane, g, [] { __syncwarp(); });
}

__device__ void warp_pair_spectra(const GreenParams& gp, double rt, double dr0, double zd,
                                  long long sid, const double* __restrict__ leg, long long n_split,
                                  const double* __restrict__ cosT, const double* __restrict__ s2T,
                                  const WarpSmem& W, int lane, const PairGrid& g) {
  const int Ms = gp.Ms, Mq = gp.Mq;
  const int nl = g.nl;  // local grid size; sample j sits at entry j of its tables
  const double* __restrict__ cosL = g.cosL;
  const int T = nl, tstride = 1;
  const int Me = g.mc + 1;  // modes 0..mc computed, the rest zero
  const int H = nl / 2 + 1, Q = nl / 4;  // samples on [0, pi]; fold point
  const double d2 = dr0 * dr0 + zd * zd;
  const double alpha = dr0 - d2 / (2.0 * rt);
  const bool split = sid >= 0;
  const cd g0 = gp.gamma0;
  warp_pair_samples(gp, rt, dr0, zd, sid, leg, n_split, cosT, W, lane, g);
  // fold: smp[j] <- w_j F_j + w_{n/2-j} F_{n/2-j} (even m), smp[n/2-j] <- difference (odd m)
  for (int t = lane; t < NFAM * Q; t += 32) {
    int f = t / Q, j = t % Q;
    cd a = W.smp[f * H + j], b = W.smp[f * H + H - 1 - j];
    W.smp[f * H + j] = a + b;
    W.smp[f * H + H - 1 - j] = a - b;
  }
  __syncwarp();
  // second fold of the even-m sums E_j (j = 0..Q, E_Q the centre sample) at
  // j <-> Q - j: cos(m phi_{Q-j}) = (-1)^{m/2} cos(m phi_j) for even m, so
  // m = 0 mod 4 sums E_j + E_{Q-j} (kept at j) over j < Q/2 plus the centre
  // E_{Q/2}, and m = 2 mod 4 sums E_j - E_{Q-j} (kept at Q - j) over j < Q/2
  // (its centre cosine vanishes).  Needs Q even (grids of 8k points).
  const int Q2 = Q / 2;
  const bool fold2 = (Q & 1) == 0;
  if (fold2) {
    for (int t = lane; t < NFAM * Q2; t += 32) {
      int f = t / Q2, j = t % Q2;
      cd a = W.smp[f * H + j], b = W.smp[f * H + Q - j];
      W.smp[f * H + j] = a + b;
      W.smp[f * H + Q - j] = a - b;
    }
    __syncwarp();
  }
  // cosine transform: spec_m = (1/n) sum_j w_j F_j cos(m phi_j) (the 4pi of G
  // is folded into the normalisation); the u^{-3/2} part is added exactly.
  const double inv = 1.0 / nl;
  const double FOUR_PI = 12.566370614359172;
  // coefficient of the exact u^{-3/2} part of family f (split pairs)
  auto beta = [&](int f) -> cd {
    switch (f) {
      case 2: case 4: return C(-alpha);
      case 3: case 5: return C(-zd);
      case 6: return (-2.0 * alpha * alpha) * g0;
      case 7: return (-2.0 * alpha * zd) * g0;
      case 8: return (-2.0 * zd * zd) * g0;
      default: return C(0.0);
    }
  };
  const double* Shat = leg + (long long)(Mq + 1) * n_split;
  // one (mode, family triple) per lane and round: 3 (M+2) items keep the
  // lanes busy where one mode per lane would leave most of the last round
  // idle.  Items run odd modes first, then m = 2 mod 4, then m = 0 mod 4
  // (with fold2), so that the lanes of a round mostly share a trip count.
  const int n_odd = Me / 2, n_2 = (Me + 1) / 4;
  for (int t = lane; t < NFAM * (Ms - Me); t += 32) W.spec[(t / (Ms - Me)) * Ms + Me + t % (Ms - Me)] = C(0.0);
  for (int it = lane; it < 3 * Me; it += 32) {
    const int k = it / 3, f0 = 3 * (it % 3);
    int mm, cls;  // cls 1: odd, 2: m = 2 mod 4, 0: m = 0 mod 4 (without fold2: 0 for every even m)
    if (!fold2) { mm = k; cls = mm & 1; }
    else if (k < n_odd) { mm = 2 * k + 1; cls = 1; }
    else if (k < n_odd + n_2) { mm = 4 * (k - n_odd) + 2; cls = 2; }
    else { mm = 4 * (k - n_odd - n_2); cls = 0; }
    cd acc[3] = {C(0.0), C(0.0), C(0.0)};
    const bool odd = cls == 1;
    const int step = (mm * tstride) % T;  // table index of cos(m phi_j) advances by step (mod T)
    const int nj = odd ? Q : (fold2 ? Q2 : Q);
    int idx = 0;
    for (int j = 0; j < nj; ++j) {
      double c = cosL[idx];
      idx += step;
      if (idx >= T) idx -= T;
      int jj = odd ? (H - 1 - j) : (cls == 2 ? Q - j : j);
#pragma unroll
      for (int f = 0; f < 3; ++f) acc[f] = fma(c, W.smp[(f0 + f) * H + jj], acc[f]);
    }
    if (cls == 0) {  // the centre sample (j = Q/2 after the second fold, else n/4) pairs with itself
      double c = cosL[idx];
      const int jc = fold2 ? Q2 : Q;
#pragma unroll
      for (int f = 0; f < 3; ++f) acc[f] = fma(c, W.smp[(f0 + f) * H + jc], acc[f]);
    }
    double Sm = split ? Shat[(long long)mm * n_split + sid] / FOUR_PI : 0.0;
#pragma unroll
    for (int f = 0; f < 3; ++f) {
      cd v = inv * acc[f];
      if (split) v = fma(Sm, beta(f0 + f), v);
      W.spec[(f0 + f) * Ms + mm] = v;
    }
  }
  __syncwarp();
}

// ---------------------------------------------------------------------------
// Stores of the Mueller 4 x 4 blocks (block.cuh forms them).
__device__ __forceinline__ void store_block(cd* __restrict__ A, int n, int m, int i, int j, cd blk[4][4],
                                            double scale) {
  size_t base = (size_t)m * n * n;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    double2* dst = (double2*)(A + base + (size_t)(4 * j + b) * n + 4 * i);
#pragma unroll
    for (int a = 0; a < 4; ++a) dst[a] = make_double2(scale * blk[a][b].x, scale * blk[a][b].y);
  }
}

__device__ __forceinline__ void store_block(cd* __restrict__ A, int n, int m, int i, int j, cd blk[4][4]) {
  size_t base = (size_t)m * n * n;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    double2* dst = (double2*)(A + base + (size_t)(4 * j + b) * n + 4 * i);
#pragma unroll
    for (int a = 0; a < 4; ++a) dst[a] = make_double2(blk[a][b].x, blk[a][b].y);
  }
}

__device__ __forceinline__ void store_zero_block(cd* __restrict__ A, int n, int m, int i, int j) {
  size_t base = (size_t)m * n * n;
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    double2* dst = (double2*)(A + base + (size_t)(4 * j + b) * n + 4 * i);
#pragma unroll
    for (int a = 0; a < 4; ++a) dst[a] = make_double2(0.0, 0.0);
  }
}

__device__ __forceinline__ bool near_panels(int Pi, int Pj, int nP, int closed) {
  int d = Pi - Pj;
  if (d >= -1 && d <= 1) return true;
  if (closed && nP > 2 && (d == nP - 1 || d == -(nP - 1))) return true;
  return false;
}

// ---------------------------------------------------------------------------
// Far panels: fused sampling, transform and assembly for one (i, j) pair per warp.
// Modes 0..M are assembled one per lane.  When M + 1 leaves a partial last
// round of tail = (M + 1) mod 32 modes (a.tq > 0), the tail modes are not
// assembled with their pair: the pair's spectra of modes full - 1 .. M + 1 go
// to a per-warp queue in global scratch, and once a.tq pairs are queued one
// round assembles all their tail blocks (a.tq * tail <= 32 lanes busy instead
// of tail lanes per pair).
__global__ void far_kernel(BuildArgs a) {
  extern __shared__ __align__(16) char smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const GreenParams& gp = a.gp;
  WarpSmem W = warp_smem(gp, smem + (size_t)wib * green_smem_bytes(gp));
  const long long total = (long long)a.N * a.N;
  const int n = 4 * a.N;
  const int tq = a.tq;
  const int full = tq ? (gp.M + 1) / 32 * 32 : gp.M + 1;  // modes assembled with their pair
  const int tail = gp.M + 1 - full, tw = tail + 2;         // queued modes, kept spectra per pair
  const long long gw = (long long)blockIdx.x * wpb + wib;
  cd* Qs = tq ? a.tailq + gw * (long long)tq * tw * NFAM : nullptr;
  int* Qij = tq ? a.tailij + gw * 2LL * tq : nullptr;
  int qn = 0;  // pairs in the queue (warp-uniform)
  // per-pair constants: quadrature weights times the L2 weight ratio, 1 / r_t
  auto pair_consts = [&](int i, int j, double fac[3], double* irt) {
    const double rs = a.geo.r[j], w = a.geo.w[j] * rs * (a.geo.sw[i] / a.geo.sw[j]);
    fac[0] = w * a.geo.rp[j];
    fac[1] = w;
    fac[2] = w * a.geo.zp[j];
    *irt = 1.0 / a.geo.r[i];
  };
  auto assemble = [&](const cd* S, int stride, int base, int i, int j, int m, const double fac[3], double irt) {
    cd blk[4][4];
    mueller_block_spec(S, stride, base, fac, m, a.ap, a.geo.r[i], irt, a.geo.rp[i], a.geo.zp[i], blk);
    store_block(a.A, n, m, i, j, blk, 1.0);
  };
  auto flush = [&]() {
    __syncwarp();  // the queue's global writes are visible to the whole warp
    for (int it = lane; it < qn * tail; it += 32) {
      const int q = it / tail, m = full + it % tail;
      double fac[3], irt;
      pair_consts(Qij[2 * q], Qij[2 * q + 1], fac, &irt);
      assemble(Qs + (long long)q * tw * NFAM, tw, full - 1, Qij[2 * q], Qij[2 * q + 1], m, fac, irt);
    }
    __syncwarp();
    qn = 0;
  };
  for (long long p = gw; p < total; p += (long long)gridDim.x * wpb) {
    int i = (int)(p / a.N), j = (int)(p % a.N);
    if (near_panels(i / P_NODES, j / P_NODES, a.n_panels, a.closed)) continue;
    long long sid = a.split_far[p];
    double rt = a.geo.r[i], rs = a.geo.r[j];
    const double dr0 = rt - rs, zd0 = a.geo.z[i] - a.geo.z[j];
    const PairGrid g = pair_grid(gp, rt, dr0, zd0, sid >= 0, a.lneps, a.cosT, a.s2T, a.ladC, a.ladS);
    warp_pair_spectra(gp, rt, dr0, zd0, sid, a.leg, a.n_split, a.cosT, a.s2T, W, lane, g);
    // modes above mz have zero spectra at m - 1, m and m + 1: their blocks are zero
    const int mz = min(gp.M, g.mc + 1);
    double fac[3], irt;
    pair_consts(i, j, fac, &irt);
    for (int m = lane; m < full; m += 32) {
      if (m <= mz) assemble(W.spec, gp.Ms, 0, i, j, m, fac, irt);
      else store_zero_block(a.A, n, m, i, j);
    }
    if (tq) {
      if (mz >= full) {
        cd* dst = Qs + (long long)qn * tw * NFAM;
        for (int t = lane; t < NFAM * tw; t += 32) dst[t] = W.spec[(t / tw) * gp.Ms + full - 1 + t % tw];
        if (lane == 0) { Qij[2 * qn] = i; Qij[2 * qn + 1] = j; }
        if (++qn == tq) flush();
      } else {
        for (int m = full + lane; m <= gp.M; m += 32) store_zero_block(a.A, n, m, i, j);
      }
    }
    __syncwarp();
  }
  if (tq && qn > 0) flush();
}

// ---------------------------------------------------------------------------
// Support points of the self and adjacent panels: one warp per
// (target, slot); spectra are written to scratch for the contraction below.
// Slot layout per target: [0, SELF_PTS) own panel, then ADJ_PTS of the
// previous panel (its shared end is +1), then ADJ_PTS of the next panel
// (shared end -1).
__device__ __forceinline__ bool support_point(const BuildArgs& a, int i, int slot, long long* pid) {
  int P = i / P_NODES, loc = i % P_NODES;
  int nP = a.n_panels;
  if (slot < SELF_PTS) {
    *pid = (long long)P * PTS_PER_PANEL + loc * SELF_PTS + slot;
    return true;
  }
  if (slot < SELF_PTS + ADJ_PTS) {
    int Q = P - 1;
    if (Q < 0) { if (!a.closed || nP <= 2) return false; Q = nP - 1; }
    if (slot - SELF_PTS >= a.sup.adj_n[2 * Q + 1]) return false;  // beyond the rule of Q's end +1
    *pid = (long long)Q * PTS_PER_PANEL + P_NODES * SELF_PTS + ADJ_PTS + (slot - SELF_PTS);
    return true;
  }
  int Q = P + 1;
  if (Q >= nP) { if (!a.closed || nP <= 2) return false; Q = 0; }
  if (slot - SELF_PTS - ADJ_PTS >= a.sup.adj_n[2 * Q + 0]) return false;  // beyond the rule of Q's end -1
  *pid = (long long)Q * PTS_PER_PANEL + P_NODES * SELF_PTS + (slot - SELF_PTS - ADJ_PTS);
  return true;
}

__global__ void support_kernel(BuildArgs a) {
  extern __shared__ __align__(16) char smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  const GreenParams& gp = a.gp;
  WarpSmem W = warp_smem(gp, smem + (size_t)wib * green_smem_bytes(gp));
  const long long total = (long long)a.N * NEAR_SLOTS;
  for (long long p = (long long)blockIdx.x * wpb + wib; p < total; p += (long long)gridDim.x * wpb) {
    int i = (int)(p / NEAR_SLOTS), slot = (int)(p % NEAR_SLOTS);
    long long pid;
    if (!support_point(a, i, slot, &pid)) continue;
    long long sid = a.split_sup[p];
    double rt = a.geo.r[i], dr0, zd;
    if (slot < SELF_PTS) { dr0 = a.sup.dr[pid]; zd = a.sup.dz[pid]; }
    else { dr0 = rt - a.sup.r[pid]; zd = a.geo.z[i] - a.sup.z[pid]; }
    const PairGrid g = pair_grid(gp, rt, dr0, zd, sid >= 0, a.lneps, a.cosT, a.s2T, a.ladC, a.ladS);
    warp_pair_spectra(gp, rt, dr0, zd, sid, a.leg, a.n_split, a.cosT, a.s2T, W, lane, g);
    cd* dst = a.spec_sup + p * NFAM * gp.Ms;
    for (int t = lane; t < NFAM * gp.Ms; t += 32) dst[t] = W.spec[t];
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
// Support spectra with the transform on the tensor cores.  The support pairs
// are sampled on the full grid (they are near pairs: their spectra keep all
// modes), and the cosine transform spec_m = (1/n) sum_j w_j F_j cos(2 pi m j / n)
// becomes one real product for a chunk of pairs: rows = (pair, family,
// Re/Im), k = j (n/2 + 1 samples), columns = modes; FP64-accurate through
// exact digit slicing (oz_real_gemm_kernel).  The sampling kernel writes each
// row's digits and scale; the product writes Y[m][row]; the last kernel forms
// the complex spectra and adds the exact u^{-3/2} part of split pairs.
#define SUP_ROWS (2 * NFAM)  // rows per pair

__device__ __forceinline__ void support_geometry(const BuildArgs& a, int i, int slot, long long pid, double* rt,
                                                 double* dr0, double* zd) {
  *rt = a.geo.r[i];
  if (slot < SELF_PTS) { *dr0 = a.sup.dr[pid]; *zd = a.sup.dz[pid]; }
  else { *dr0 = *rt - a.sup.r[pid]; *zd = a.geo.z[i] - a.sup.z[pid]; }
}

// ---------------------------------------------------------------------------
// Geometry and tables of a build, formed on the device (on the host they took
// 2 to 4 ms per body: thread starts, N^2 flags uploaded, one copy per table).

// cosines and sin^2 of every grid: blockIdx.y = 0 the full grid, q the ladder grid of 8 q points
__global__ void tables_kernel(int nphi, int qmax, double* __restrict__ tab) {
  const int q = blockIdx.y, t = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = q ? 8 * q : nphi;
  if (q == 1 || t >= n) return;  // the ladder starts at 16 points
  double *c = tab, *s2 = tab + nphi;
  if (q) {
    double* lad = tab + nphi + nphi / 2 + 1;
    c = lad + (4 * (q - 1) * q - 8);
    s2 = lad + ladder_cos_doubles(qmax) + (2 * (q - 1) * q - 4 + (q - 2));
  }
  c[t] = cospi(2.0 * t / n);
  if (t <= n / 2) {
    const double v = sinpi((double)t / n);
    s2[t] = v * v;
  }
}

// one thread per support point: geometry from the panel's degree-15 interpolants
__global__ void __launch_bounds__(128) support_points_kernel(BuildArgs a, const double* __restrict__ ndr,
                                                             const double* __restrict__ ndz,
                                                             const double* __restrict__ wt_self,
                                                             const double* __restrict__ wt_adj,
                                                             double* __restrict__ sup) {
  const int t = blockIdx.x * 128 + threadIdx.x, Q = blockIdx.y;
  if (t >= PTS_PER_PANEL) return;
  const size_t npts = (size_t)a.n_panels * PTS_PER_PANEL, id = (size_t)Q * PTS_PER_PANEL + t;
  const bool own = t < P_NODES * SELF_PTS;
  const double* L = nullptr;
  double wt = 0.0;
  if (own) {
    L = a.sup.Lself + (size_t)t * P_NODES;
    wt = wt_self[t];
  } else {
    const int e = (t - P_NODES * SELF_PTS) / ADJ_PTS, s = (t - P_NODES * SELF_PTS) % ADJ_PTS;
    const int rule = a.sup.adj_rule[2 * Q + e];
    if (rule >= 0 && s < a.sup.adj_n[2 * Q + e]) {
      const size_t k = (size_t)(rule * 2 + e) * ADJ_PTS + s;
      L = a.sup.Ladj + k * P_NODES;
      wt = wt_adj[k];
    }
  }
  double v[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (L) {  // else no neighbour at this end, or beyond the rule's points
    const double *r = a.geo.r + Q * P_NODES, *z = a.geo.z + Q * P_NODES;
    const double *dr = ndr + Q * P_NODES, *dz = ndz + Q * P_NODES;
    double vr = 0.0, vz = 0.0, vdr = 0.0, vdz = 0.0, ddr = 0.0, ddz = 0.0;
    const int tgt = own ? t / SELF_PTS : -1;
    for (int k = 0; k < P_NODES; ++k) {
      vr += L[k] * r[k]; vz += L[k] * z[k]; vdr += L[k] * dr[k]; vdz += L[k] * dz[k];
      if (own && k != tgt) {  // x_t - x_s = -sum_{k != t} L_k(tau_s) (x_k - x_t)
        ddr -= L[k] * (r[k] - r[tgt]);
        ddz -= L[k] * (z[k] - z[tgt]);
      }
    }
    const double sp = hypot(vdr, vdz);
    v[0] = vr; v[1] = vz; v[2] = vdr / sp; v[3] = vdz / sp; v[4] = wt * sp; v[5] = ddr; v[6] = ddz;
  }
#pragma unroll
  for (int f = 0; f < 7; ++f) sup[f * npts + id] = v[f];
}

// One warp per target: COUNT the split pairs of its row, or number and list them
// in order of source and slot from the rows' prefix sums.
template <bool COUNT>
__global__ void __launch_bounds__(128) split_rows_kernel(BuildArgs a, double cthr, int* __restrict__ row,
                                                         int* __restrict__ split_far, int* __restrict__ split_sup,
                                                         double* __restrict__ pairs, int* __restrict__ sup_list) {
  const int i = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= a.N) return;
  const double rt = a.geo.r[i], zt = a.geo.z[i];
  int nf = COUNT ? 0 : row[i], ns = COUNT ? 0 : row[a.N + i], nv = COUNT ? 0 : row[2 * a.N + i];
  const unsigned below = (1u << lane) - 1u;
  auto put = [&](int id, double dr, double dz) {
    double* v = pairs + 4 * (size_t)id;
    v[0] = rt; v[1] = zt; v[2] = dr; v[3] = dz;
  };
  for (int j0 = 0; j0 < a.N; j0 += 32) {  // N is a multiple of 16
    const int j = j0 + lane;
    const bool far = j < a.N && !near_panels(i / P_NODES, j / P_NODES, a.n_panels, a.closed);
    const double dr = far ? rt - a.geo.r[j] : 0.0, dz = far ? zt - a.geo.z[j] : 0.0;
    const bool sp = far && split_pair(rt, dr, dz, cthr);
    const unsigned b = __ballot_sync(0xffffffffu, sp);
    if (!COUNT && j < a.N) {
      const int id = nf + __popc(b & below);
      split_far[(size_t)i * a.N + j] = sp ? id : -1;
      if (sp) put(id, dr, dz);
    }
    nf += __popc(b);
  }
  for (int s0 = 0; s0 < NEAR_SLOTS; s0 += 32) {  // a multiple of 32
    const int slot = s0 + lane;
    long long pid = 0;
    const bool ok = support_point(a, i, slot, &pid);
    double r, dr = 0.0, dz = 0.0;
    if (ok) support_geometry(a, i, slot, pid, &r, &dr, &dz);
    const bool sp = ok && split_pair(rt, dr, dz, cthr);
    const unsigned b = __ballot_sync(0xffffffffu, sp), v = __ballot_sync(0xffffffffu, ok);
    if (!COUNT) {
      const int id = ns + __popc(b & below);
      split_sup[(size_t)i * NEAR_SLOTS + slot] = sp ? id : -1;
      if (sp) put(id, dr, dz);
      if (ok) sup_list[nv + __popc(v & below)] = i * NEAR_SLOTS + slot;
    }
    ns += __popc(b);
    nv += __popc(v);
  }
  if (COUNT && lane == 0) { row[i] = nf; row[a.N + i] = ns; row[2 * a.N + i] = nv; }
}

// Exclusive prefix sum of `count` integers in place (one CTA of 1024); returns the total.
__device__ int block_scan(int* __restrict__ v, long long count, int* part) {
  const long long per = (count + 1023) / 1024, lo = min(count, threadIdx.x * per), hi = min(count, lo + per);
  int sum = 0;
  for (long long k = lo; k < hi; ++k) sum += v[k];
  __syncthreads();
  part[threadIdx.x] = sum;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int x = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
    __syncthreads();
    part[threadIdx.x] += x;
    __syncthreads();
  }
  int run = part[threadIdx.x] - sum;
  for (long long k = lo; k < hi; ++k) {
    const int x = v[k];
    v[k] = run;
    run += x;
  }
  __syncthreads();
  return part[1023];
}

__global__ void __launch_bounds__(1024) split_scan_kernel(int* __restrict__ row, int N, int* __restrict__ counts) {
  __shared__ int part[1024];
  const int split = block_scan(row, 2LL * N, part);
  const int pts = block_scan(row + 2 * N, N, part);
  if (threadIdx.x == 0) { counts[0] = split; counts[1] = pts; }
}

void launch_tables(const GreenParams& gp, double* tab, cudaStream_t s) {
  tables_kernel<<<dim3((gp.nphi + 127) / 128, gp.qmax >= 2 ? gp.qmax + 1 : 1), 128, 0, s>>>(gp.nphi, gp.qmax, tab);
}

void launch_support_points(const BuildArgs& a, const double* dr, const double* dz, const double* wt_self,
                           const double* wt_adj, double* sup, cudaStream_t s) {
  support_points_kernel<<<dim3((PTS_PER_PANEL + 127) / 128, a.n_panels), 128, 0, s>>>(a, dr, dz, wt_self, wt_adj, sup);
}

void launch_split_count(const BuildArgs& a, double cthr, int* row, int* counts, cudaStream_t s) {
  split_rows_kernel<true><<<(a.N + 3) / 4, 128, 0, s>>>(a, cthr, row, nullptr, nullptr, nullptr, nullptr);
  split_scan_kernel<<<1, 1024, 0, s>>>(row, a.N, counts);
}

void launch_split_list(const BuildArgs& a, double cthr, const int* row, int* split_far, int* split_sup,
                       double* pairs, int* sup_list, cudaStream_t s) {
  split_rows_kernel<false><<<(a.N + 3) / 4, 128, 0, s>>>(a, cthr, const_cast<int*>(row), split_far, split_sup, pairs,
                                                         sup_list);
}

// CTA of SUP_NT threads per support pair of the chunk: list[q0 + q], q < count.
// Shared: the samples [NFAM][H], q [H], the Legendre coefficients [Mq + 1].
#define SUP_NT 128

__host__ __device__ inline int support_sample_smem(int H, int Mq) {
  return NFAM * H * 16 + H * 8 + (Mq + 1) * 8 + (SUP_NT / 32) * SUP_ROWS * 8 + SUP_ROWS * 8;
}

// Row scales and digits of one pair's samples W.smp[f][j], j < H, as rows
// q * 18 + (2 f + Re/Im) of the digit operand (k-tiles of 16, nkt of them):
// by the SUP_NT threads of the CTA.
__device__ __forceinline__ void pair_rows_to_digits(const WarpSmem& W, int H, int q, int nkt,
                                                    __nv_bfloat16* __restrict__ Asl, double* __restrict__ Ascale,
                                                    double* red, double* shift) {
  const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
  // row maxima of |v| on the bits of the samples (integer pipe)
  unsigned long long mx[SUP_ROWS];
#pragma unroll
  for (int rr = 0; rr < SUP_ROWS; ++rr) mx[rr] = 0ull;
  for (int j = t; j < H; j += SUP_NT)
#pragma unroll
    for (int f = 0; f < NFAM; ++f) {
      const cd v = W.smp[f * H + j];
      const unsigned long long bx = abs_bits(v.x), by = abs_bits(v.y);
      mx[2 * f] = bx > mx[2 * f] ? bx : mx[2 * f];
      mx[2 * f + 1] = by > mx[2 * f + 1] ? by : mx[2 * f + 1];
    }
#pragma unroll
  for (int rr = 0; rr < SUP_ROWS; ++rr) {
    unsigned long long m = mx[rr];
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long y = __shfl_xor_sync(0xffffffffu, m, o);
      m = y > m ? y : m;
    }
    if (lane == 0) red[wid * SUP_ROWS + rr] = __longlong_as_double((long long)m);
  }
  __syncthreads();
  if (t < SUP_ROWS) {  // row scales: powers of two 2^E above twice each row's largest magnitude
    double m = 0.0;
    for (int w = 0; w < SUP_NT / 32; ++w) m = fmax(m, red[w * SUP_ROWS + t]);
    const int E = pow2_scale_exp(m);
    shift[t] = (double)(56 - E);  // digits of round(v 2^(56 - E))
    Ascale[(size_t)q * SUP_ROWS + t] = ldexp(1.0, E);
  }
  __syncthreads();
  // digits: thread item = (row, group of 8 consecutive k), one 16-byte store per digit
  const int kg_n = nkt * 2;
  for (int it = t; it < SUP_ROWS * kg_n; it += SUP_NT) {
    const int rr = it / kg_n, kg = it % kg_n, f = rr >> 1, im = rr & 1;
    const int S = (int)shift[rr];
    int dg[8][OZ_S];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const int k = kg * 8 + c;
      double v = 0.0;
      if (k < H) { const cd z = W.smp[f * H + k]; v = im ? z.y : z.x; }
      digits28(fixed_rn(v, S), dg[c]);
    }
    const long long row = (long long)q * SUP_ROWS + rr;
    const long long rt_ = row >> 7;
    const int r = (int)(row & 127), kt = kg >> 1, kk = (kg & 1) * 8;
    __nv_bfloat16* blk = Asl + ((size_t)rt_ * nkt + kt) * (OZ_S * 2048);
    const int off = core_off(r, kk);
#pragma unroll
    for (int d = 0; d < OZ_S; ++d) {
      __align__(16) __nv_bfloat16 e8[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) e8[c] = __float2bfloat16((float)dg[c][d]);
      *(uint4*)(blk + d * 2048 + off) = *(uint4*)e8;
    }
  }
  __syncthreads();  // the shared samples are rewritten by the next pair
}

__device__ __forceinline__ WarpSmem sample_smem(char* smem, int H, int Mq, double** red, double** shift) {
  WarpSmem W;
  W.smp = (cd*)smem;
  W.spec = nullptr;
  W.q = (double*)(W.smp + NFAM * H);
  W.phs = W.q + H;
  *red = W.phs + Mq + 1;                // [SUP_NT / 32][SUP_ROWS]
  *shift = *red + (SUP_NT / 32) * SUP_ROWS;  // [SUP_ROWS]
  return W;
}

// FAR: the pairs are far pairs (p = i N + j) on the full grid, else support
// pairs (p = i NEAR_SLOTS + slot).
template <int RR, bool FAR>
__global__ void __launch_bounds__(SUP_NT, 3) support_sample_kernel(BuildArgs a, const int* __restrict__ list, int q0,
                                                                   int count, __nv_bfloat16* __restrict__ Asl,
                                                                   double* __restrict__ Ascale, int nkt) {
  extern __shared__ __align__(16) char smem[];
  const GreenParams& gp = a.gp;
  double *red, *shift;
  const WarpSmem W = sample_smem(smem, gp.H, gp.Mq, &red, &shift);
  for (int q = blockIdx.x; q < count; q += gridDim.x) {
    const int p = list[q0 + q];
    double rt, dr0, zd;
    long long sid;
    if (FAR) {
      const int i = p / a.N, j = p % a.N;
      rt = a.geo.r[i];
      dr0 = rt - a.geo.r[j];
      zd = a.geo.z[i] - a.geo.z[j];
      sid = a.split_far[p];
    } else {
      const int i = p / NEAR_SLOTS, slot = p % NEAR_SLOTS;
      long long pid;
      support_point(a, i, slot, &pid);
      support_geometry(a, i, slot, pid, &rt, &dr0, &zd);
      sid = a.split_sup[p];
    }
    group_pair_samples<SUP_NT, RR>(gp, rt, dr0, zd, sid, a.leg, a.n_split, a.cosT, W, threadIdx.x,
                                   full_grid(gp, a.cosT, a.s2T), [] { __syncthreads(); });
    __syncthreads();
    pair_rows_to_digits(W, gp.H, q, nkt, Asl, Ascale, red, shift);
  }
}

// Far pairs of one bin below the full grid (list[q0 + q], q < count, p = i N + j;
// never split) on their ladder grid of nl points: the same rows as the support
// pairs.  A CTA takes PB pairs at a time and deals out (pair, sample) items, so
// that grids of 9 to 129 samples fill its warps; the bin's grid is known, only
// its table is looked up.
__host__ __device__ inline int far_sample_smem_per_pair(int H) { return NFAM * H * 16 + SUP_ROWS * 4; }

template <int RR>
__global__ void __launch_bounds__(128, 4) far_sample_kernel(BuildArgs a, const int* __restrict__ list, int q0, int count,
                                                            __nv_bfloat16* __restrict__ Asl,
                                                            double* __restrict__ Ascale, int nkt, int nl, int PB) {
  extern __shared__ __align__(16) char smem[];
  const GreenParams& gp = a.gp;
  const int H = nl / 2 + 1, tid = threadIdx.x, qq = nl / 8;
  const double* __restrict__ s2L = a.ladS + (2 * (qq - 1) * qq - 4 + (qq - 2));  // see pair_grid
  cd* smp = (cd*)smem;                       // [PB][NFAM][H]
  int* shift = (int*)(smp + (size_t)PB * NFAM * H);  // [PB][SUP_ROWS]
  for (long long b0 = (long long)blockIdx.x * PB; b0 < count; b0 += (long long)gridDim.x * PB) {
    const int np = (int)min((long long)PB, count - b0);
    for (int it = tid; it < np * H; it += 128) {
      const int q = it / H, j = it - q * H;
      const int p = list[q0 + b0 + q], i = p / a.N, jn = p % a.N;
      const double rt = a.geo.r[i], rs = a.geo.r[jn];
      PairSample ps;
      ps.dr0 = rt - rs;
      ps.zd = a.geo.z[i] - a.geo.z[jn];
      ps.d2 = ps.dr0 * ps.dr0 + ps.zd * ps.zd;
      ps.rr4 = 4.0 * rt * rs;
      ps.rs2 = 2.0 * rs;
      ps.irt = ps.alpha = 0.0;
      const double w = (j == 0 || j == H - 1) ? 0.5 : 1.0;
      pair_sample<RR >= 1, RR == 2>(gp, ps, s2L[j], w, false, 0.0, smp + (size_t)q * NFAM * H + j, H);
    }
    __syncthreads();
    // row scales: powers of two 2^E above twice each row's largest magnitude, on
    // the bits of the samples; four threads per row
    for (int t0 = 0; t0 < np * SUP_ROWS * 4; t0 += 128) {
      const int t = t0 + tid, rw = t >> 2, q = rw / SUP_ROWS, rr = rw - q * SUP_ROWS;
      unsigned long long mx = 0ull;
      if (rw < np * SUP_ROWS) {
        const double* x = (const double*)(smp + ((size_t)q * NFAM + (rr >> 1)) * H) + (rr & 1);
        for (int j = t & 3; j < H; j += 4) {
          const unsigned long long b = abs_bits(x[2 * j]);
          mx = b > mx ? b : mx;
        }
      }
      for (int o = 2; o > 0; o >>= 1) {
        const unsigned long long y = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = y > mx ? y : mx;
      }
      if ((t & 3) == 0 && rw < np * SUP_ROWS) {
        const int E = pow2_scale_exp(__longlong_as_double((long long)mx));
        shift[rw] = 56 - E;  // digits of round(v 2^(56 - E))
        Ascale[(size_t)b0 * SUP_ROWS + rw] = ldexp(1.0, E);
      }
    }
    __syncthreads();
    const int kg_n = nkt * 2;
    for (int it = tid; it < np * SUP_ROWS * kg_n; it += 128) {
      const int rw = it / kg_n, kg = it - rw * kg_n, q = rw / SUP_ROWS, rr = rw - q * SUP_ROWS;
      const double* x = (const double*)(smp + ((size_t)q * NFAM + (rr >> 1)) * H) + (rr & 1);
      const int S = shift[rw];
      int dg[8][OZ_S];
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const int k = kg * 8 + c;
        digits28(k < H ? fixed_rn(x[2 * k], S) : 0ll, dg[c]);
      }
      const long long row = b0 * SUP_ROWS + rw;
      __nv_bfloat16* blk = Asl + ((size_t)(row >> 7) * nkt + (kg >> 1)) * (OZ_S * 2048) +
                           core_off((int)(row & 127), (kg & 1) * 8);
#pragma unroll
      for (int d = 0; d < OZ_S; ++d) {
        __align__(16) __nv_bfloat16 e8[8];
#pragma unroll
        for (int c = 0; c < 8; ++c) e8[c] = __float2bfloat16((float)dg[c][d]);
        *(uint4*)(blk + d * 2048) = *(uint4*)e8;
      }
    }
    __syncthreads();  // the samples are rewritten by the next pairs
  }
}

// Far pairs listed bin by bin (bin: g.nl / 8), within a bin by source j and then
// by target i up to a tile of FAR_TILE pairs, so that pairs assembled together
// write the same columns side by side and the order does not depend on timing
// beyond a tile.  tag[j N + i] packs the bin and the highest mode m_c (7 and 9 bits:
// n_phi is at most 512 on this path); 0xFFFF marks near pairs.
// tile_hist[bin][tile]: pairs of each bin in each tile of the (j, i) order.
#define FAR_TILE 1024
#define FAR_NEAR 0xFFFF
static_assert((OZR_KMAX - 1) * 2 / 8 < 127 && OZR_KMAX < 511, "bin and mode fit the tag");
__global__ void __launch_bounds__(256) far_bin_kernel(BuildArgs a, unsigned short* __restrict__ tag, int nbins,
                                                      int ntiles, int* __restrict__ tile_hist) {
  extern __shared__ int hist[];
  for (int b = threadIdx.x; b < nbins; b += 256) hist[b] = 0;
  __syncthreads();
  const GreenParams& gp = a.gp;
  for (int t = threadIdx.x; t < FAR_TILE; t += 256) {
    const long long p = (long long)blockIdx.x * FAR_TILE + t;  // j N + i
    if (p >= (long long)a.N * a.N) break;
    const int j = (int)(p / a.N), i = (int)(p % a.N);
    if (near_panels(i / P_NODES, j / P_NODES, a.n_panels, a.closed)) { tag[p] = FAR_NEAR; continue; }
    const double rt = a.geo.r[i], dr0 = rt - a.geo.r[j], zd0 = a.geo.z[i] - a.geo.z[j];
    const PairGrid g = pair_grid(gp, rt, dr0, zd0, a.split_far[(long long)i * a.N + j] >= 0, a.lneps, a.cosT, a.s2T,
                                 a.ladC, a.ladS);
    const int b = g.nl / 8;
    tag[p] = (unsigned short)(b << 9 | g.mc);
    atomicAdd(&hist[b], 1);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < nbins; b += 256) tile_hist[(size_t)b * ntiles + blockIdx.x] = hist[b];
}

// Prefix sums of the tiles' counts and each bin's start (start[nbins]: the total).
__global__ void __launch_bounds__(1024) far_scan_kernel(int* __restrict__ v, long long count, int nbins, int ntiles,
                                                        int* __restrict__ start) {
  __shared__ int part[1024];
  const int total = block_scan(v, count, part);
  for (int b = threadIdx.x; b < nbins; b += 1024) start[b] = v[(size_t)b * ntiles];
  if (threadIdx.x == 0) start[nbins] = total;
}

__global__ void __launch_bounds__(256) far_scatter_kernel(int N, const unsigned short* __restrict__ tag, int nbins,
                                                          int ntiles, const int* __restrict__ tile_start,
                                                          int* __restrict__ list, unsigned short* __restrict__ mcs) {
  extern __shared__ int cursor[];
  for (int b = threadIdx.x; b < nbins; b += 256) cursor[b] = tile_start[(size_t)b * ntiles + blockIdx.x];
  __syncthreads();
  for (int t = threadIdx.x; t < FAR_TILE; t += 256) {
    const long long p = (long long)blockIdx.x * FAR_TILE + t;
    if (p >= (long long)N * N) break;
    const int b = tag[p];
    if (b == FAR_NEAR) continue;
    const int q = atomicAdd(&cursor[b >> 9], 1);
    list[q] = (int)(p % N) * N + (int)(p / N);
    mcs[q] = (unsigned short)(b & 511);
  }
}

// The blocks of far pairs from their spectra Y[m][row] (the products of one
// bin's chunk): modes above the pair's m_c zero, the split pairs' u^{-3/2} part
// added, the families of block.cuh combined once per pair and mode in shared
// memory, then one block per (pair, mode) and thread.  A CTA takes PB pairs of
// the bin at a time, so that (pair, mode) items fill its lanes whatever the
// bin's number of modes.  FP64 pipe, 40 % busy (the rest barriers and latency):
// N = 1024, M = 128 64 -> 50 ms, the cylinder (lossy) 19.5 -> 9.8 ms, against a warp
// per pair with the block formed from the nine spectra.
struct FarPair {
  double irt, rpt, zpt, h0, h1, f2;  // target, weights (1 / nl in them)
  double alpha, zd;                      // u^{-3/2} part of a split pair
  int i, j, Me, mz, sid;                 // nodes, computed modes, last mode with a block, split id
};

template <bool SIMPLE>
__global__ void __launch_bounds__(128) far_assemble_kernel(BuildArgs a, const int* __restrict__ list,
                                                           const unsigned short* __restrict__ mcs, int q0, int count,
                                                           const double* __restrict__ Y, int ldy, int ncols, int nl,
                                                           int PB) {
  extern __shared__ __align__(16) char smem[];
  const GreenParams& gp = a.gp;
  const int W = ncols + 2;               // modes 0..ncols + 1 of a pair's families
  cd* comb = (cd*)smem;                  // [PB][BK_N][W]
  FarPair* pp = (FarPair*)(comb + (size_t)PB * BK_N * W);
  const int tid = threadIdx.x, n = 4 * a.N;
  const int mmax = min(gp.M, ncols);     // blocks above are zero for every pair of the bin
  const bool unit = a.ap.aEJ.x == 1.0 && a.ap.aEJ.y == 0.0 && a.ap.aHM.x == -1.0 && a.ap.aHM.y == 0.0;
  const double* Shat = a.leg + (long long)(gp.Mq + 1) * a.n_split;
  const double invn = 1.0 / nl;
  for (long long b0 = (long long)blockIdx.x * PB; b0 < count; b0 += (long long)gridDim.x * PB) {
    const int np = (int)min((long long)PB, count - b0);
    if (tid < np) {  // no division or logarithm here: the other threads wait for it
      const int p = list[q0 + b0 + tid];
      FarPair v;
      v.i = p / a.N;
      v.j = p % a.N;
      v.sid = a.split_far[p];
      v.irt = a.geo.irt[v.i];
      v.rpt = a.geo.rp[v.i];
      v.zpt = a.geo.zp[v.i];
      const int mc = mcs[q0 + b0 + tid];
      v.Me = min(mc + 1, ncols);
      v.mz = min(gp.M, mc + 1);
      v.alpha = v.zd = 0.0;
      if (v.sid >= 0) {
        const double rt = a.geo.r[v.i], dr0 = rt - a.geo.r[v.j];
        v.zd = a.geo.z[v.i] - a.geo.z[v.j];
        v.alpha = dr0 - (dr0 * dr0 + v.zd * v.zd) / (2.0 * rt);
      }
      const double w = a.geo.wr[v.j] * a.geo.sw[v.i] * invn;
      v.h0 = 0.5 * w * a.geo.rp[v.j];
      v.h1 = 0.5 * w;
      v.f2 = w * a.geo.zp[v.j];
      pp[tid] = v;
    }
    __syncthreads();
    for (int it = tid; it < np * W; it += 128) {
      const int q = it / W, m = it - q * W;
      const FarPair& v = pp[q];
      cd* o = comb + (size_t)q * BK_N * W + m;
      if (m >= v.Me) {
#pragma unroll
        for (int f = 0; f < BK_N; ++f) o[f * W] = C(0.0);
        continue;
      }
      const double2* y = (const double2*)(Y + (size_t)m * ldy + (b0 + q) * SUP_ROWS);  // even offset: 16-byte aligned
      cd S[NFAM];
#pragma unroll
      for (int f = 0; f < NFAM; ++f) {
        const double2 t = y[f];
        S[f] = C(t.x, t.y);
      }
      if (v.sid >= 0) {
        const double Sm = Shat[(long long)m * a.n_split + v.sid] / 12.566370614359172 * nl;
        const double al = Sm * v.alpha, zd = Sm * v.zd;
        S[2].x -= al; S[4].x -= al;
        S[3].x -= zd; S[5].x -= zd;
        S[6] = fma(-2.0 * al * v.alpha, gp.gamma0, S[6]);
        S[7] = fma(-2.0 * al * v.zd, gp.gamma0, S[7]);
        S[8] = fma(-2.0 * zd * v.zd, gp.gamma0, S[8]);
      }
      mueller_combine<SIMPLE>(S, a.ap, v.irt, v.rpt, v.zpt, o, W);
    }
    __syncthreads();
    for (int it = tid; it < np * (mmax + 1); it += 128) {
      const int q = it / (mmax + 1), m = it - q * (mmax + 1);
      const FarPair& v = pp[q];
      if (m > v.mz) { store_zero_block(a.A, n, m, v.i, v.j); continue; }
      cd blk[4][4];
      mueller_block_combined(comb + (size_t)q * BK_N * W, W, m, a.ap, unit, v.h0, v.h1, v.f2, v.irt, v.rpt, v.zpt, blk);
      store_block(a.A, n, m, v.i, v.j, blk);
    }
    const int nz = gp.M - mmax;
    for (int it = tid; it < np * nz; it += 128) {
      const int q = it / nz, m = mmax + 1 + it % nz;
      store_zero_block(a.A, n, m, pp[q].i, pp[q].j);
    }
    __syncthreads();
  }
}

// thread per (pair q, family f, mode m): spec = (1/n)(Y_re + i Y_im) + the
// exact u^{-3/2} part of a split pair (its coefficient beta_f and S^_m)
__global__ void support_post_kernel(BuildArgs a, const int* __restrict__ list, int q0, int count,
                                    const double* __restrict__ Y, int ldy) {
  const GreenParams& gp = a.gp;
  const int Ms = gp.Ms;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)count * NFAM * Ms) return;
  const int m = (int)(t % Ms);
  const int f = (int)((t / Ms) % NFAM);
  const int q = (int)(t / ((long long)Ms * NFAM));
  const int p = list[q0 + q];
  const long long row = (long long)q * SUP_ROWS + 2 * f;
  const double invn = 1.0 / gp.nphi;
  cd v = C(invn * Y[(size_t)m * ldy + row], invn * Y[(size_t)m * ldy + row + 1]);
  const long long sid = a.split_sup[p];
  if (sid >= 0 && f >= 2) {
    const int i = p / NEAR_SLOTS, slot = p % NEAR_SLOTS;
    long long pid;
    support_point(a, i, slot, &pid);
    double rt, dr0, zd;
    support_geometry(a, i, slot, pid, &rt, &dr0, &zd);
    const double d2 = dr0 * dr0 + zd * zd;
    const double alpha = dr0 - d2 / (2.0 * rt);
    const cd g0 = gp.gamma0;
    cd beta;
    switch (f) {
      case 2: case 4: beta = C(-alpha); break;
      case 3: case 5: beta = C(-zd); break;
      case 6: beta = (-2.0 * alpha * alpha) * g0; break;
      case 7: beta = (-2.0 * alpha * zd) * g0; break;
      default: beta = (-2.0 * zd * zd) * g0; break;
    }
    const double* Shat = a.leg + (long long)(gp.Mq + 1) * a.n_split;
    const double Sm = Shat[(long long)m * a.n_split + sid] / 12.566370614359172;  // / 4 pi
    v = fma(Sm, beta, v);
  }
  a.spec_sup[(size_t)p * NFAM * Ms + (size_t)f * Ms + m] = v;
}

// ---------------------------------------------------------------------------
// Near panels: R_k(sigma, f, m) = sum_s W_s L_k(tau_s) sigma_s F_f(s, m)
// (eqs. eq_nyslike, eq_nyslike2 with sum_j U_jk P_j = L_k), then the blocks of
// the panel's columns k.  One CTA per (target, near panel, chunk of kc columns).
__global__ void __launch_bounds__(384) near_kernel(BuildArgs a) {
  extern __shared__ __align__(16) char smem[];
  const GreenParams& gp = a.gp;
  const int kc = a.kc, nchunk = P_NODES / kc;
  int bid = blockIdx.x;
  const int chunk = bid % nchunk; bid /= nchunk;
  const int which = bid % 3;  // 0 prev, 1 self, 2 next
  const int i = bid / 3;
  const int P = i / P_NODES, loc = i % P_NODES, nP = a.n_panels;
  int Q, slot0, S;
  const double* L;
  if (which == 1) {
    Q = P; slot0 = 0; S = SELF_PTS; L = a.sup.Lself + (size_t)loc * SELF_PTS * P_NODES;
  } else if (which == 0) {  // previous panel: its end +1 touches the target's panel
    Q = P - 1;
    if (Q < 0) { if (!a.closed || nP <= 2) return; Q = nP - 1; }
    slot0 = SELF_PTS; S = a.sup.adj_n[2 * Q + 1];
    L = a.sup.Ladj + (size_t)(a.sup.adj_rule[2 * Q + 1] * 2 + 1) * ADJ_PTS * P_NODES;
  } else {                  // next panel: its end -1
    Q = P + 1;
    if (Q >= nP) { if (!a.closed || nP <= 2) return; Q = 0; }
    slot0 = SELF_PTS + ADJ_PTS; S = a.sup.adj_n[2 * Q + 0];
    L = a.sup.Ladj + (size_t)(a.sup.adj_rule[2 * Q + 0] * 2 + 0) * ADJ_PTS * P_NODES;
  }
  const int Ms = gp.Ms;
  cd* R = (cd*)smem;                              // [kc][3][NFAM][Ms]
  double* V = (double*)(R + (size_t)kc * 3 * NFAM * Ms);  // [S][kc][3]
  for (int t = threadIdx.x; t < S * kc; t += blockDim.x) {
    int s = t / kc, kk = t % kc;
    long long pid;
    support_point(a, i, slot0 + s, &pid);
    double w = a.sup.W[pid] * L[(size_t)s * P_NODES + chunk * kc + kk];
    double rs = a.sup.r[pid];
    V[(s * kc + kk) * 3 + 0] = w * rs * a.sup.rp[pid];
    V[(s * kc + kk) * 3 + 1] = w * rs;
    V[(s * kc + kk) * 3 + 2] = w * rs * a.sup.zp[pid];
  }
  __syncthreads();
  const cd* F = a.spec_sup + ((long long)i * NEAR_SLOTS + slot0) * NFAM * Ms;
  for (int item = threadIdx.x; item < NFAM * Ms; item += blockDim.x) {
    cd acc[8][3];
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
#pragma unroll
      for (int sg = 0; sg < 3; ++sg) acc[kk][sg] = C(0.0);
    for (int s = 0; s < S; ++s) {
      cd v = F[(size_t)s * NFAM * Ms + item];
      const double* Vs = V + s * kc * 3;
#pragma unroll
      for (int kk = 0; kk < 8; ++kk) {
        if (kk < kc) {
#pragma unroll
          for (int sg = 0; sg < 3; ++sg) acc[kk][sg] = fma(Vs[kk * 3 + sg], v, acc[kk][sg]);
        }
      }
    }
#pragma unroll
    for (int kk = 0; kk < 8; ++kk)
      if (kk < kc)
#pragma unroll
        for (int sg = 0; sg < 3; ++sg) R[((size_t)kk * 3 + sg) * NFAM * Ms + item] = acc[kk][sg];
  }
  __syncthreads();
  const int n = 4 * a.N;
  const double rt = a.geo.r[i], rpt = a.geo.rp[i], zpt = a.geo.zp[i];
  for (int item = threadIdx.x; item < kc * (gp.M + 1); item += blockDim.x) {
    int kk = item / (gp.M + 1), m = item % (gp.M + 1);
    int j = Q * P_NODES + chunk * kc + kk;
    const cd* Rk = R + (size_t)kk * 3 * NFAM * Ms;
    auto Rget = [&](int s, int f, int mm) { return Rk[((size_t)s * NFAM + f) * Ms + mm]; };
    cd blk[4][4];
    mueller_block(Rget, m, a.ap, rt, rpt, zpt, blk);
    if (j == i) {
      blk[0][2] += a.ap.dEM; blk[1][3] += a.ap.dEM;
      blk[2][0] += a.ap.dHJ; blk[3][1] += a.ap.dHJ;
    }
    store_block(a.A, n, m, i, j, blk, a.geo.sw[i] / a.geo.sw[j]);
  }
}

// ---------------------------------------------------------------------------
// Stand-alone spectra of arbitrary pairs (used by the modal-kernel entry point).
__global__ void pair_spectra_kernel(GreenParams gp, const double* __restrict__ pairs, const int* __restrict__ sidx,
                                    const double* __restrict__ leg, long long n_split, long long npairs,
                                    const double* __restrict__ cosT, const double* __restrict__ s2T,
                                    cd* __restrict__ out) {
  extern __shared__ __align__(16) char smem[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = blockDim.x >> 5;
  WarpSmem W = warp_smem(gp, smem + (size_t)wib * green_smem_bytes(gp));
  for (long long p = (long long)blockIdx.x * wpb + wib; p < npairs; p += (long long)gridDim.x * wpb) {
    const double* q = pairs + 4 * p;  // (r_t, z_t, r_t - r_s, z_t - z_s)
    warp_pair_spectra(gp, q[0], q[2], q[3], sidx[p], leg, n_split, cosT, s2T, W, lane, full_grid(gp, cosT, s2T));
    cd* dst = out + p * NFAM * gp.Ms;
    for (int t = lane; t < NFAM * gp.Ms; t += 32) dst[t] = W.spec[t];
    __syncwarp();
  }
}

// ---------------------------------------------------------------------------
static int warps_per_block(const GreenParams& gp) {
  int per = green_smem_bytes(gp);
  int w = (200 * 1024) / per;
  if (w > 8) w = 8;
  if (w < 1) w = 1;
  return w;
}

bool green_fits_smem(const GreenParams& gp) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess || optin <= 0)
    optin = 227 * 1024;
  return green_smem_bytes(gp) <= optin;
}

static int grid_for(long long units, int wpb) {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long need = (units + wpb - 1) / wpb;
  long long cap = (long long)sms * 8;
  return (int)(need < cap ? need : cap);
}

// Tail queue of far_kernel: pairs per flush (0 = none) and its scratch, for
// the launch shape launch_far_assembly uses.
int far_tail_pairs(const GreenParams& gp) {
  const int full = (gp.M + 1) / 32 * 32, tail = gp.M + 1 - full;
  return (full >= 32 && tail > 0 && tail <= 16) ? 32 / tail : 0;
}

size_t far_tail_scratch(const BuildArgs& a, size_t* ij_elems) {
  const int tq = far_tail_pairs(a.gp);
  const int wpb = warps_per_block(a.gp);
  const long long total = (long long)a.N * a.N;
  const long long warps = (long long)grid_for(total, wpb) * wpb;
  const int tail = a.gp.M + 1 - (a.gp.M + 1) / 32 * 32;
  *ij_elems = tq ? (size_t)warps * 2 * tq : 0;
  return tq ? (size_t)warps * tq * (tail + 2) * NFAM : 0;
}

void launch_far_assembly(const BuildArgs& a, cudaStream_t s) {
  int wpb = warps_per_block(a.gp);
  int smem = wpb * green_smem_bytes(a.gp);
  smem_optin(far_kernel);
  far_kernel<<<grid_for((long long)a.N * a.N, wpb), wpb * 32, smem, s>>>(a);
}

void launch_support_spectra(const BuildArgs& a, cudaStream_t s) {
  int wpb = warps_per_block(a.gp);
  int smem = wpb * green_smem_bytes(a.gp);
  smem_optin(support_kernel);
  support_kernel<<<grid_for((long long)a.N * NEAR_SLOTS, wpb), wpb * 32, smem, s>>>(a);
}

template <int RR, bool FAR>
static void launch_full_samples(const BuildArgs& a, const int* list, int q0, int count, __nv_bfloat16* Asl,
                                double* Ascale, int nkt, cudaStream_t s) {
  const int smem = support_sample_smem(a.gp.H, a.gp.Mq);
  smem_optin(support_sample_kernel<RR, FAR>);
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int grid = std::min(count, 3 * sms * 8);
  support_sample_kernel<RR, FAR><<<grid, SUP_NT, smem, s>>>(a, list, q0, count, Asl, Ascale, nkt);
}

void launch_support_samples(const BuildArgs& a, const int* list, int q0, int count, __nv_bfloat16* Asl,
                            double* Ascale, int nkt, cudaStream_t s) {
  if (a.gp.k0_real && a.gp.k1_real) launch_full_samples<2, false>(a, list, q0, count, Asl, Ascale, nkt, s);
  else if (a.gp.k0_real) launch_full_samples<1, false>(a, list, q0, count, Asl, Ascale, nkt, s);
  else launch_full_samples<0, false>(a, list, q0, count, Asl, Ascale, nkt, s);
}

int far_tiles(int N) { return (int)(((long long)N * N + FAR_TILE - 1) / FAR_TILE); }

void launch_far_bins(const BuildArgs& a, int nbins, unsigned short* tag, int* tile_hist, int* start,
                     cudaStream_t s) {
  const int tiles = far_tiles(a.N);
  far_bin_kernel<<<tiles, 256, nbins * sizeof(int), s>>>(a, tag, nbins, tiles, tile_hist);
  far_scan_kernel<<<1, 1024, 0, s>>>(tile_hist, (long long)nbins * tiles, nbins, tiles, start);
}

void launch_far_scatter(int N, int nbins, const unsigned short* tag, const int* tile_start, int* list,
                        unsigned short* mcs, cudaStream_t s) {
  far_scatter_kernel<<<far_tiles(N), 256, nbins * sizeof(int), s>>>(N, tag, nbins, far_tiles(N), tile_start, list, mcs);
}

// Pairs per CTA: among those that leave four CTAs per SM (registers; 54 KiB of
// shared memory each), the number whose (pair, sample) items waste the fewest
// lanes; one pair of the largest ladder grid takes 19 KiB.
template <int RR>
static void launch_ladder_samples(const BuildArgs& a, const int* list, int q0, int count, __nv_bfloat16* Asl,
                                  double* Ascale, int nkt, int nl, cudaStream_t s) {
  const int H = nl / 2 + 1, per = far_sample_smem_per_pair(H);
  int PB = 1;
  double best = 0.0;
  for (int b = 1; b <= 32 && (b == 1 || b * per <= 54 * 1024); ++b) {
    const double eff = (double)b * H / ((b * H + 127) / 128 * 128);
    if (eff > best + 0.02) { best = eff; PB = b; }
  }
  smem_optin(far_sample_kernel<RR>);
  far_sample_kernel<RR><<<grid_for(count, PB), 128, PB * per, s>>>(a, list, q0, count, Asl, Ascale, nkt, nl, PB);
}

template <int RR>
static void launch_far_samples_rr(const BuildArgs& a, const int* list, int q0, int count, __nv_bfloat16* Asl,
                                  double* Ascale, int nkt, int nl, cudaStream_t s) {
  if (nl == a.gp.nphi) launch_full_samples<RR, true>(a, list, q0, count, Asl, Ascale, nkt, s);
  else launch_ladder_samples<RR>(a, list, q0, count, Asl, Ascale, nkt, nl, s);
}

void launch_far_samples(const BuildArgs& a, const int* list, int q0, int count, __nv_bfloat16* Asl, double* Ascale,
                        int nkt, int nl, cudaStream_t s) {
  if (a.gp.k0_real && a.gp.k1_real) launch_far_samples_rr<2>(a, list, q0, count, Asl, Ascale, nkt, nl, s);
  else if (a.gp.k0_real) launch_far_samples_rr<1>(a, list, q0, count, Asl, Ascale, nkt, nl, s);
  else launch_far_samples_rr<0>(a, list, q0, count, Asl, Ascale, nkt, nl, s);
}

// Pairs per CTA: among those that leave four CTAs per SM (registers; 56 KiB of
// shared memory each), the number whose (pair, mode) items waste the fewest lanes
// of the last round; at least one, whatever it takes of shared memory.
void launch_far_assemble(const BuildArgs& a, const int* list, const unsigned short* mcs, int q0, int count,
                         const double* Y, int ldy, int ncols, int nl, cudaStream_t s) {
  const int per = BK_N * (ncols + 2) * 16 + (int)sizeof(FarPair), items = std::min(a.gp.M, ncols) + 1;
  int PB = 1;
  double best = 0.0;
  for (int b = 1; b <= 32 && (b == 1 || b * per <= 56 * 1024); ++b) {
    const double eff = (double)b * items / ((b * items + 127) / 128 * 128);
    if (eff > best + 0.02) { best = eff; PB = b; }
  }
  const int smem = PB * per, grid = grid_for(count, PB);
  if (a.ap.simple) {
    smem_optin(far_assemble_kernel<true>);
    far_assemble_kernel<true><<<grid, 128, smem, s>>>(a, list, mcs, q0, count, Y, ldy, ncols, nl, PB);
  } else {
    smem_optin(far_assemble_kernel<false>);
    far_assemble_kernel<false><<<grid, 128, smem, s>>>(a, list, mcs, q0, count, Y, ldy, ncols, nl, PB);
  }
}

void launch_support_post(const BuildArgs& a, const int* list, int q0, int count, const double* Y, int ldy,
                         cudaStream_t s) {
  const long long items = (long long)count * NFAM * a.gp.Ms;
  support_post_kernel<<<(unsigned)((items + 255) / 256), 256, 0, s>>>(a, list, q0, count, Y, ldy);
}

// Threads per CTA: the fewest rounds (at most 384 threads) over the larger
// of the contraction's NFAM (M+2) items and the kc (M+1) blocks, so that the
// last round is not nearly empty (one CTA per SM: its shared memory).
void launch_near_assembly(const BuildArgs& a, cudaStream_t s) {
  int smem = a.kc * 3 * NFAM * a.gp.Ms * 16 + NEAR_MAX_PTS * a.kc * 3 * 8;
  const int items = std::max(NFAM * a.gp.Ms, a.kc * (a.gp.M + 1));
  const int rounds = (items + 383) / 384;
  const int threads = std::min(384, ((items + rounds - 1) / rounds + 31) / 32 * 32);
  smem_optin(near_kernel);
  near_kernel<<<a.N * 3 * (P_NODES / a.kc), threads, smem, s>>>(a);
}

void launch_pair_spectra(const GreenParams& gp, const double* pairs, const int* sidx, const double* leg,
                         long long n_split, long long npairs, const double* cosT, const double* s2T, cd* out,
                         cudaStream_t s) {
  if (npairs <= 0) return;
  int wpb = warps_per_block(gp);
  int smem = wpb * green_smem_bytes(gp);
  smem_optin(pair_spectra_kernel);
  pair_spectra_kernel<<<grid_for(npairs, wpb), wpb * 32, smem, s>>>(gp, pairs, sidx, leg, n_split, npairs, cosT,
                                                                      s2T, out);
}

// ---------------------------------------------------------------------------
// Allocation-free variant of mueller_modal_kernels (declared in mueller.h).
// Its scratch (transform tables, split flags, pair displacements, Laplace-type
// coefficients) lives in one fixed file-scope device array instead of memory
// from cudaMalloc.  Host code must not use the array's name as a device
// address: its address is fetched once per device with cudaGetSymbolAddress.
#include <mutex>
#include "mueller.h"

#define NOALLOC_SCRATCH_DOUBLES ((size_t)2 * 1024 * 1024)  // 16 MiB
static __device__ __align__(256) double g_noalloc_scratch[NOALLOC_SCRATCH_DOUBLES];

#define NOALLOC_MAX_DEVICES 64
// Per-device set-up state, written under g_noalloc_mu: the scratch array's
// device address and whether the series tables were uploaded to that device.
static std::mutex g_noalloc_mu;
static double* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {nullptr};
static bool g_noalloc_tables[NOALLOC_MAX_DEVICES] = {false};
// message reported by mueller_last_error (defined with the other ABI functions)
void mueller_internal_set_error(const char* msg);

__global__ void noalloc_tables_kernel(int nphi, double* __restrict__ cosT, double* __restrict__ s2T) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < nphi) cosT[t] = cospi(2.0 * t / nphi);
  if (t <= nphi / 2) {
    double v = sinpi((double)t / nphi);
    s2T[t] = v * v;
  }
}

// (r_t, z_t, r_s, z_s) -> (r_t, z_t, r_t - r_s, z_t - z_s); split flag per pair
__global__ void noalloc_prep_kernel(const double* __restrict__ pairs, long long n, int nphi, int M, double lneps,
                                    double* __restrict__ disp, int* __restrict__ sid) {
  long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= n) return;
  double rt = pairs[4 * p], zt = pairs[4 * p + 1];
  double dr = rt - pairs[4 * p + 2], dz = zt - pairs[4 * p + 3];
  disp[4 * p] = rt; disp[4 * p + 1] = zt; disp[4 * p + 2] = dr; disp[4 * p + 3] = dz;
  double d2 = dr * dr + dz * dz, B = 2.0 * rt * (rt - dr);
  double c = d2 / B, cp1 = 2.0 + c;
  double lz = log1p(c + sqrt(c * cp1));
  sid[p] = ((double)(nphi - M - 1) * lz < lneps) ? (int)p : -1;
}

__global__ void noalloc_legendre_kernel(const double* __restrict__ disp, const int* __restrict__ sid, long long n,
                                        int Mq, int Ms, double* __restrict__ leg, int nr) {
  extern __shared__ double rinv[];
  fill_odd_reciprocals(rinv, nr);
  long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (p >= n || sid[p] < 0) return;
  legendre_one(disp[4 * p], disp[4 * p + 2], disp[4 * p + 3], p, n, Mq, Ms, leg, rinv, nr);
}

static int noalloc_fail(const char* msg, int code = MUELLER_EINVAL) {
  mueller_internal_set_error(msg);
  return code;
}

extern "C" int mueller_modal_kernels_noalloc(const double* pairs_dev, long long npairs, mueller_c128 k0,
                                             mueller_c128 k1, int M, int n_phi, double split_eps,
                                             mueller_c128* out_dev, void* stream) {
  mueller_internal_set_error("");
  if (!pairs_dev || !out_dev || npairs < 0 || M < 0) return noalloc_fail("invalid arguments");
  if (n_phi < 16 || n_phi > 8192 || (n_phi & (n_phi - 1)) != 0) return noalloc_fail("n_phi must be a power of two in [16, 8192]");
  if (M + 2 > n_phi / 2) return noalloc_fail("n_phi must be at least 2M + 4");
  if (k0.im < 0 || k1.im < 0) return noalloc_fail("wavenumbers need Im k >= 0");
  if (npairs == 0) return MUELLER_OK;
  const int Mq = n_phi / 2 - 1, Ms = M + 2, H = n_phi / 2 + 1;
  {
    GreenParams g{};
    g.Ms = Ms; g.H = H; g.Mq = Mq;
    if (!green_fits_smem(g)) return noalloc_fail("n_phi and M need more shared memory per warp than a CTA can have");
  }
  auto up32 = [](size_t v) { return (v + 31) & ~(size_t)31; };
  const size_t o_cos = 0, o_s2 = o_cos + up32(n_phi), o_disp = o_s2 + up32(H);
  const size_t o_sid = o_disp + up32(4 * (size_t)npairs);
  const size_t o_leg = o_sid + up32(((size_t)npairs + 1) / 2);
  const size_t need = o_leg + (size_t)(Mq + 1 + Ms) * (size_t)npairs;
  if (need > NOALLOC_SCRATCH_DOUBLES) {
    char msg[200];
    snprintf(msg, sizeof(msg), "npairs * (n_phi/2 + M + 7) exceeds the fixed scratch of %zu doubles (16 MiB): need %zu",
             (size_t)NOALLOC_SCRATCH_DOUBLES, need);
    return noalloc_fail(msg);
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return noalloc_fail("no current CUDA device");
  double* base = nullptr;
  {  // one-time set-up on this device (host threads serialised)
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      double* p = nullptr;
      cudaError_t e = cudaGetSymbolAddress((void**)&p, g_noalloc_scratch);
      if (e != cudaSuccess || !p) return noalloc_fail(cudaGetErrorString(e), MUELLER_ECUDA);
      g_noalloc_ptr[dev] = p;
    }
    if (!g_noalloc_tables[dev]) {
      SeriesTables t;
      fill_series_tables(&t);
      if (cudaMemcpyToSymbol(c_tab, &t, sizeof(SeriesTables)) != cudaSuccess) return noalloc_fail("series tables");
      g_noalloc_tables[dev] = true;
    }
    base = g_noalloc_ptr[dev];
  }
  double* cosT = base + o_cos;
  double* s2T = base + o_s2;
  double* disp = base + o_disp;
  int* sid = (int*)(base + o_sid);
  double* leg = base + o_leg;
  cudaStream_t s = (cudaStream_t)stream;
  GreenParams gp{};
  cd K0{k0.re, k0.im}, K1{k1.re, k1.im};
  gp.M = M; gp.Ms = Ms; gp.nphi = n_phi; gp.H = H; gp.Mq = Mq; gp.qmax = 0;
  gp.kp0 = kpow(K0); gp.kp1 = kpow(K1);
  gp.gamma0 = -0.25 * (K0 * K0 - K1 * K1);
  gp.k0_real = K0.y == 0.0; gp.k1_real = K1.y == 0.0;
  double eps = split_eps > 0 ? split_eps : 1e-17;
  noalloc_tables_kernel<<<(n_phi + 255) / 256, 256, 0, s>>>(n_phi, cosT, s2T);
  unsigned blocks = (unsigned)((npairs + 127) / 128);
  noalloc_prep_kernel<<<blocks, 128, 0, s>>>(pairs_dev, npairs, n_phi, M, -log(eps), disp, sid);
  const int nr = legendre_table_entries(Mq);
  smem_optin(noalloc_legendre_kernel);
  noalloc_legendre_kernel<<<blocks, 128, nr * 8, s>>>(disp, sid, npairs, Mq, Ms, leg, nr);
  launch_pair_spectra(gp, disp, sid, leg, npairs, npairs, cosT, s2T, (cd*)out_dev, s);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return noalloc_fail(cudaGetErrorString(e), MUELLER_ECUDA);
  return MUELLER_OK;
}
