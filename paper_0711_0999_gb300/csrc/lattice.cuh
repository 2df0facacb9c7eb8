// Internal launchers of the lattice-step kernels (not part of the C ABI).
#pragma once

#include "common.cuh"

namespace nedmft {

int launch_build_s(const ContourDev& c, const double2* sigma, double2* S, cudaStream_t st);
int launch_g0_build(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, int nq,
                    double2* g0, cudaStream_t st);
int launch_gen_a(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, int q0, int nb,
                 const double2* S, double2* A, int np, cudaStream_t st);

// Largest n_c of the single-CTA FP64 Gauss-Jordan path (whole matrix in shared memory).
constexpr int kSmallPathMaxN = 112;
int small_path_max_n();
int launch_gj_small_fp64(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, int q0,
                         int nb, const double2* S, double2* out, int* status, cudaStream_t st);

// Element (i, j) of an np x np matrix of the FP64 tensor-core path: boxes of 32 rows x 8 columns, 4 KB each and
// row-band major, so that the update adds a box by one contiguous bulk reduction; within a box a row's 128 bytes
// with the columns exchanged by the row's low bits, the order in which a lane per row writes a box to shared memory
// without bank conflicts.  Eight columns of a row from a multiple of 8 on stay one 128-byte line.
__host__ __device__ __forceinline__ size_t box_off(int np, int i, int j) {
  return ((size_t)(i >> 5) * (np >> 3) + (j >> 3)) * 256 + (i & 31) * 8 + ((j ^ i) & 7);
}

// Batched FP64 inverses on the tensor cores (gj64_umma.cu): nb matrices of np x np in that order (np a multiple of
// 128, the identity outside n x n), in place, scratch of gj64_scratch_bytes.
size_t gj64_scratch_bytes(int np, int nb);
int gj64_invert(double2* A, int n, int np, int nb, void* scratch, int* status, cudaStream_t st);
int gj64_set_wait_ns(uint64_t ns, cudaStream_t st);  // its bounded waits' limit on the current device

int launch_reduce(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, const double* wq,
                  int q0, int nb, const double2* X, int ldx, bool cycled, bool first, double2* gloc, double2* jacc,
                  cudaStream_t st);
int launch_finish_current(int nt, const double2* jacc, double* j, double* ji, cudaStream_t st);

// Dense FP64 inversion with partial pivoting (impurity step).
size_t pivot_inverse_workspace(int n);
int pivot_inverse(double2* a, int n, void* ws, cudaStream_t st, int* status);
int pivot_inverse_prepare();  // before capturing pivot_inverse into a graph

}  // namespace nedmft
