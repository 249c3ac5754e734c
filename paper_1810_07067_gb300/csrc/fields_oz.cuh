// Far field on a grid: the product of ring integrals and currents on the tensor
// cores (fields_oz.cu), and the far-field vector both forms of that product end in.
#pragma once
#include <cuda_bf16.h>
#include "cplx.cuh"
#include "fields.cuh"
#include "fields_plan.cuh"

// F of mode m (index q) at polar angle p and, when it is another one, at its mirror
// n_polar - 1 - p, from the sums A (cosine of the phase) and B (sine): u = 0, 1, 2
// of J1/J2 and then of M1/M2 (see ffgrid_mode_kernel); dst is F[w].
__device__ __forceinline__ void ffgrid_vector(const cd* A, const cd* B, int m, int M, double k0, double omega, cd eps0,
                                              int p, int n_polar, cd* dst) {
  const int mi[3] = {abs(m + 1), abs(m), abs(m - 1)};
  double sth, cth;
  sincospi((p + 0.5) / n_polar, &sth, &cth);
  const double inv4pi = 1.0 / (4.0 * 3.141592653589793);
  const cd pre = -C(k0 * k0) / (C(0.0, omega) * eps0);
  const cd ik = C(0.0, k0);
  for (int mir = 0; mir < 2; ++mir) {
    const int pm = mir ? n_polar - 1 - p : p;
    if (mir && pm == p) break;
    const double c = mir ? -cth : cth;
    cd t[6];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      cd U[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const cd iB = mul_i(B[3 * h + u]);
        cd v = mir ? A[3 * h + u] - iB : A[3 * h + u] + iB;
        U[u] = (mi[u] & 1) ? -mul_i(v) : v;  // c_m = -i b_m for odd m
      }
      t[3 * h] = 0.5 * (U[0] + U[2]);
      t[3 * h + 1] = -mul_i(0.5 * (U[0] - U[2]));
      t[3 * h + 2] = U[1];
    }
    const double xh[3] = {sth, 0.0, c};
    const cd xJ = xh[0] * t[0] + xh[2] * t[2];
    cd cr[3];
    cr[0] = xh[1] * t[5] - xh[2] * t[4];
    cr[1] = xh[2] * t[3] - xh[0] * t[5];
    cr[2] = xh[0] * t[4] - xh[1] * t[3];
    cd* o = dst + ((size_t)pm * (2 * M + 1) + (m + M)) * 3;
    for (int a = 0; a < 3; ++a) o[a] = inv4pi * (pre * (t[a] - xh[a] * xJ) + ik * cr[a]);
  }
}

// The whole grid by products on the tensor cores: ring integrals, sums over the nodes
// (into F), sums over the modes (into E); work of plan.bytes (256-byte aligned), plan the
// ffo_plan of the same arguments; err (device int) is set if a bounded wait gives up.
void launch_ffgrid_products(const FieldGeom& g, int M, double k0, double omega, cd eps0, const cd* x, int nrhs,
                            int n_polar, int n_azim, int n_alpha, const FfoPlan& plan, void* work, cd* F, cd* E, int* err,
                            cudaStream_t s);

// Modal data of the waves w0 .. w0 + count - 1 (count <= RHS_WAVES) of nrhs from their
// table (rhs_wave_kernel without the factors fE, fH of the traces); work of plan.bytes
// (256-byte aligned), plan the rhs_plan of the same nrhs.
void launch_rhs_products(const FieldGeom& g, int M, const double2* wave, const cd* tab, cd fE, cd fH, int w0, int count,
                         int nrhs, int n_theta, const RhsPlan& plan, void* work, cd* rhs, int* err, cudaStream_t s);

// Fields of nrhs right-hand sides at nt points from their ring points and currents
// (ring_kernel) into out[w][p][6]; work of plan.bytes (256-byte aligned), plan the
// nf_plan of the same points and at least as many sides.
void launch_nearfield_products(long long total, const double4* pts, const cd* cur, const double* X, int nt, int nrhs,
                               cd k, cd cJ, cd cM, cd dM, cd dJ, const NfPlan& plan, void* work, cd* out, int* err,
                               cudaStream_t s);
