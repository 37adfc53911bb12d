// Launch interface of the fixed-point multipole-to-local translations
// (mc_m2l.cu).
#pragma once
#include <cuda_runtime.h>
#include <stddef.h>

// the matrices of every offset up to signs, for order p: one device table of
// this size, filled from a scratch of 2 x 343 (2p+1)(p+1) doubles
size_t m2l_table_bytes(int p);
cudaError_t m2l_build_table(int p, int sms, void* table, double* otab, cudaStream_t st);
// chunks of the offsets per target that fill the SMs on a level with nl cells
// per axis (scratch: cells x chunks x C doubles when above 1)
int m2l_chunks(int nl, int sms);
// Lout = translations of the multipoles K of level l (cell width w) over the
// interaction lists; M, E: cells x C and cells integers of workspace
cudaError_t m2l_fix_level(int p, int l, double w, bool pbc, int sms, const void* table, const double* K, long long* M,
                          int* E, double* Lout, double* scratch, size_t scratch_doubles, cudaStream_t st);
