// Products of the complex128 LU on BF16 tensor cores (see lu_oz.cu).
#pragma once
#include <cuda_runtime.h>
#include "lu.cuh"

#define ZB 128  // columns of an outer block (four LU_NB panels) = largest inner dimension

// Workspace bytes of one n x n matrix (LuMat::ws, 256-byte aligned).
size_t luz_matrix_bytes(int n);

// Before the first panel: the exponents of the matrices' columns.
void luz_begin(const LuMat* d, int nmax, int count, cudaStream_t s);
// Rows k0..k0+LU_NB of U in the `cols` columns of the block right of the panel.
void luz_panel_rows(const LuMat* d, int K0, int k0, int cols, int count, cudaStream_t s);
// C = A[k0+LU_NB.., k0+LU_NB..min(K0+ZB, n)) -= L U of the panel at column k0 of the
// block at K0, for the first `count` matrices of the table (nmax the largest n).
int luz_panel_update(const LuMat* d, int K0, int k0, int nmax, int count, int* err, cudaStream_t s);
// Columns right of the block at K0 (interchanges applied): U = L11^{-1} A12,
// then A22 -= L21 U.  For matrices with n > K0 + ZB.  Both return their launches.
int luz_block_update(const LuMat* d, int K0, int nmax, int count, int* err, cudaStream_t s);
