// FP64 H.X from integer-slice products on the tensor cores (sliced_hx.cu; internal).
#pragma once

#include <cuda_runtime.h>

#include <cstddef>

#include "hx_kernels.cuh"

namespace cs {

struct HostTables;

// set-up tables of one basis, and W V of the current potential, as integer slices
struct SlicedTables {
  unsigned char* tab[6] = {};  // digit images of the six contractions' tables
  int* exps = nullptr;         // table-row exponents: R1, then R2, L2 and the radial scaling
  size_t off_f2 = 0, off_fl = 0, off_re = 0;
  int F1 = 0;                  // exponent of the Legendre table of the synthesis
  long long* wv = nullptr;     // [k][j][q] W V below the row's power of two
  int* ewv = nullptr;          // [k][j]
};

// lmax <= 62, n_theta <= 128, n_phi <= 255 (64 table rows or K per class); N, n_r <= 448 (the
// 64-bit sums of the radial products)
bool sliced_hx_eligible(int L, int N, int n_r, int n_theta, int n_phi);
// whether CS_ANGULAR_KERNEL leaves them on (df: for a double-float call)
bool sliced_hx_enabled(bool df);
// default size of the chunk intermediates
constexpr size_t kSlChunkBytes = (size_t)512 << 20;
size_t sliced_hx_work_bytes(int L, int n_r, int n_theta, int n_phi, int S);
// A smaller workspace for S states: the fixed part and intermediates of at least one radial node.
// The results do not depend on the split: every scale belongs to one state's row.
size_t sliced_hx_fixed_bytes(int n_r, int S);
size_t sliced_hx_node_bytes(int L, int n_theta, int n_phi, int S);
// rad, theta: the FP64 device tables
cudaError_t build_sliced_tables(const HostTables& H, const double* rad, const double* theta,
                                SlicedTables& T);
void free_sliced_tables(SlicedTables& T);
cudaError_t launch_sliced_wv(const SlicedTables& T, const double* wv, int rows, int n_phi,
                             cudaStream_t st);
// stage 0: radial synthesis X -> G; 1: the angular block on G, in place; 2: radial analysis of G
// with the epilogue. *launches receives the kernel count. bytes: room for the chunk intermediates.
cudaError_t launch_sliced_hx(const HostTables& H, const SlicedTables& T, int S, const double* X,
                             long long ld, double* G, const Epilogue<double>& ep, void* work,
                             int* err, cudaStream_t st, int stage, int* launches,
                             size_t bytes = kSlChunkBytes);

// Grid values f[s][k][j][q] of S columns of X, or, with X null, of the radial synthesis in G.
cudaError_t launch_sliced_grid(const HostTables& H, const SlicedTables& T, int S, const double* X,
                               long long ld, double* G, double* f, void* work, int* err,
                               cudaStream_t st, int* launches);
// rho (+)= 2 sum_s occ[s] f[s]^2, in state order
cudaError_t launch_sliced_density(const HostTables& H, const SlicedTables& T, int S,
                                  const double* X, long long ld, const double* occ, bool add,
                                  double* G, double* rho, void* work, int* err, cudaStream_t st,
                                  int* launches);
// Analysis of S grid functions g[s][k][j][q] times the row weights wkj, with the epilogue.
cudaError_t launch_sliced_forward(const HostTables& H, const SlicedTables& T, int S,
                                  const double* g, const double* wkj, double* G,
                                  const Epilogue<double>& ep, void* work, int* err,
                                  cudaStream_t st, int* launches);

}  // namespace cs
