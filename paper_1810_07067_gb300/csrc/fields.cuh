#pragma once
#include <cuda_runtime.h>
#include "cplx.cuh"

struct FieldGeom {
  const double *r, *z, *rp, *zp, *w;  // nodes [N]
  int N;
};

// Modal plane-wave data: rhs[q][w][4N], q = m + M (k0 real, n_theta a multiple
// of 4); scratch of rhs_planewave_scratch_doubles values, 16-byte aligned, and work
// of rhs_planewave_work_bytes (256-byte aligned; null: the ring integrals run on the
// FP64 pipe); err (device int) is set if a bounded wait gives up.  False, with nothing
// launched, when work_bytes do not hold the layout.
size_t rhs_planewave_scratch_doubles(int M, int nrhs, int n_theta);
size_t rhs_planewave_work_bytes(int N, int M, int nrhs, int n_theta);
bool launch_rhs_planewave(const FieldGeom& g, int M, double k0, double omega, cd mu0, cd sE, cd sH,
                          const double* dirs_dev, const double* pols_dev, int nrhs, int n_theta, double* scratch,
                          void* work, size_t work_bytes, cd* rhs, int* err, cudaStream_t s);

// Far field E[rhs][dir][3] from currents x[q][rhs][4N]; ring work buffer
// cur[rhs][N][n_theta][4].
void launch_far_field(const FieldGeom& g, int M, cd k0, double omega, cd eps0, const cd* x, int nrhs,
                      const double* dirs_dev, int ndir, int n_theta, cd* cur, cd* E, cudaStream_t s);

// Modal data from sampled incident fields EH[rhs][N][n_theta][6] (device).
void launch_rhs_samples(const FieldGeom& g, int M, cd sE, cd sH, const cd* EH, int nrhs, int n_theta, cd* rhs,
                        cudaStream_t s);

// E, H at points X[nt][3] (device) into out[rhs][nt][6], gr = near_field_group
// right-hand sides at a time; work buffers cur [gr][N][n_theta][6], pts
// [N][n_theta][4] (32-byte aligned), and either work of near_field_work_bytes
// (256-byte aligned; err, a device int, is set if a bounded wait gives up) or part of
// near_field_part values (work null: FP64 pipe); k and the four constants are the
// region's.  total = N n_theta, a multiple of 16.  False, with nothing launched, when
// work_bytes do not hold the layout.
int near_field_group(long long total, int nrhs);
size_t near_field_work_bytes(long long total, int nt, int nrhs);
size_t near_field_part(long long total, int nt, int nrhs);
bool launch_near_field(const FieldGeom& g, int M, const cd* x, int nrhs, const double* X_dev, int nt, int n_theta,
                       cd k, cd cJ, cd cM, cd dM, cd dJ, cd* cur, double* pts, cd* part, void* work, size_t work_bytes,
                       cd* out, int* err, cudaStream_t s);

// Far field on the grid theta_p = (p + 1/2) pi / n_polar, phi_s = 2 pi s / n_azim:
// E[rhs][p][s][3] (k0 real, n_alpha a multiple of 4); F [rhs][n_polar][2M+1][3] and
// either work of far_field_grid_work_bytes (256-byte aligned; err, a device int, is
// set if a bounded wait gives up) or coef of far_field_grid_coef_doubles values (work
// null: FP64 pipe).  False, with nothing launched, when work_bytes do not hold the layout.
size_t far_field_grid_coef_doubles(int N, int M, int n_polar);
size_t far_field_grid_work_bytes(int N, int M, int n_polar, int n_azim, int n_alpha, int nrhs);
bool launch_far_field_grid(const FieldGeom& g, int M, double k0, double omega, cd eps0, const cd* x, int nrhs,
                           int n_polar, int n_azim, int n_alpha, double* coef, void* work, size_t work_bytes, cd* F, cd* E,
                           int* err, cudaStream_t s);

// Currents x[v][n] at the nodes -> xs[v][4 nsub] at refined nodes (rows Lm[nsub][16]
// of the panel interpolants, node0 = first node of each sub-node's panel).
void launch_interp_currents(const cd* x, int n, int nsub, const int* node0, const double* Lm, long long nvec, cd* xs,
                            cudaStream_t s);
