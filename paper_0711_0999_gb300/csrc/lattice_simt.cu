// CUDA-core kernels of the lattice step: S = W Sigma W, the dense G0 builder,
// the FP64 path's B_q - S generator, Gauss-Jordan inversion of small matrices
// in shared memory (a CTA per point) and the FP64 quadrature / current
// reductions.
#include "lattice.cuh"

namespace nedmft {

// ------------------------------------------------------------------ S = W Sigma W

__global__ void build_s_kernel(ContourDev c, const double2* __restrict__ sigma, double2* __restrict__ S) {
  size_t total = (size_t)c.n * c.n;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(e / c.n), j = (int)(e % c.n);
    S[e] = cmul(cmul(weight(c, i), sigma[e]), weight(c, j));
  }
}

int launch_build_s(const ContourDev& c, const double2* sigma, double2* S, cudaStream_t st) {
  size_t total = (size_t)c.n * c.n;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 152 * 16) blocks = 152 * 16;
  build_s_kernel<<<blocks, 256, 0, st>>>(c, sigma, S);
  NED_LAUNCH_CHECK("build_s_kernel");
  return NEDMFT_OK;
}

// ------------------------------------------------------------------ G0 (dense)

// G0(t_i, t_j) of Eq. g_contour_non_final2 in the log-stable form:
//   i >= j: -i exp(-x (tau_i - tau_j) - softplus(-beta x)) e^{i phase},
//   i <  j:  i exp(-x (tau_i - tau_j) - softplus( beta x)) e^{i phase},
// phase = mu Re(t_i - t_j) - [F(t_i) - F(t_j)].
__global__ void g0_build_kernel(ContourDev c, ModelDev m, const double* __restrict__ eps_d,
                                const double* __restrict__ ebar_d, double2* __restrict__ g0) {
  const int q = blockIdx.y;
  const double eps = eps_d[q], ebar = ebar_d[q];
  const double x = eps - m.mu;
  const double sp_neg = x > 0 ? log1p(exp(-c.beta * x)) : -c.beta * x + log1p(exp(c.beta * x));   // softplus(-beta x)
  const double sp_pos = x > 0 ? c.beta * x + log1p(exp(-c.beta * x)) : log1p(exp(c.beta * x));    // softplus(beta x)
  size_t total = (size_t)c.n * c.n;
  double2* out = g0 + (size_t)q * total;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    int i = (int)(e / c.n), j = (int)(e % c.n);
    double si = t_re(c, i), sj = t_re(c, j);
    double ph = m.mu * (si - sj) - band_phase_diff(sj, si, eps, ebar, m.E);
    double re = -x * (t_tau(c, i) - t_tau(c, j));
    double sn, cs;
    sincos(ph, &sn, &cs);
    double mag, pre;
    if (i >= j) { mag = exp(re - sp_neg); pre = -1.0; } else { mag = exp(re - sp_pos); pre = 1.0; }
    // pre * i * mag * (cs + i sn) = pre * mag * (-sn + i cs)
    out[e] = make_double2(-pre * mag * sn, pre * mag * cs);
  }
}

int launch_g0_build(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, int nq,
                    double2* g0, cudaStream_t st) {
  size_t total = (size_t)c.n * c.n;
  int bx = (int)((total + 255) / 256);
  if (bx > 1024) bx = 1024;
  dim3 grid(bx, nq);
  g0_build_kernel<<<grid, 256, 0, st>>>(c, m, eps, ebar, g0);
  NED_LAUNCH_CHECK("g0_build_kernel");
  return NEDMFT_OK;
}

// ------------------------------------------------------------------ A'_q = P (B_q - S), padded

// 32 rows of one matrix per CTA: the first warp forms the rows' entries of B_q
// (one lane per row, so a sincos and an exponential per row run side by side),
// then a warp per row copies -S and adds them.  One pass over the output: HBM
// bound.  (With the entry of B_q formed where the copying thread met it, one
// lane of a warp ran that chain while 31 waited: 450 us for 100 matrices of
// 256 x 256, 105 MB.)
constexpr int kGenRows = 32;
__global__ void __launch_bounds__(256) gen_a_kernel(ContourDev c, ModelDev m, const double* __restrict__ eps_d,
                                                    const double* __restrict__ ebar_d, int q0,
                                                    const double2* __restrict__ S, double2* __restrict__ A, int np) {
  const int r0 = blockIdx.x * kGenRows, b = blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __shared__ double2 sub[kGenRows];  // the entry of B_q left of the diagonal, or in the corner for row 0
  __shared__ int src_row[kGenRows];
  if (warp == 0) {
    const double eps = eps_d[q0 + b], ebar = ebar_d[q0 + b];
    const int r = r0 + lane;
    int i = r;
    if (r < c.n && shifted_point(m, eps)) i = r + 1 == c.n ? 0 : r + 1;
    src_row[lane] = i;
    if (i < c.n) sub[lane] = i >= 1 ? b_sub(c, m, eps, ebar, i) : b_corner(c, m, eps);
  }
  __syncthreads();
  for (int rr = warp; rr < kGenRows; rr += 8) {
    const int i = src_row[rr];
    double2* dst = A + (size_t)b * np * np;
    const int r = r0 + rr;
    if (i >= c.n) {  // padding
      for (int j = lane; j < np; j += 32) dst[box_off(np, r, j)] = make_double2(j == i ? 1.0 : 0.0, 0.0);
      continue;
    }
    const double2* src = S + (size_t)i * c.n;
    const int js = i >= 1 ? i - 1 : c.n - 1;
    for (int j = lane; j < np; j += 32) {
      double2 v = make_double2(0.0, 0.0);
      if (j < c.n) {
        v = src[j];
        v.x = -v.x;
        v.y = -v.y;
        if (j == i) v.y += 1.0;
        if (j == js) v = cadd(v, sub[rr]);
      }
      dst[box_off(np, r, j)] = v;
    }
  }
}

int launch_gen_a(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, int q0, int nb,
                 const double2* S, double2* A, int np, cudaStream_t st) {
  gen_a_kernel<<<dim3(np / kGenRows, nb), 256, 0, st>>>(c, m, eps, ebar, q0, S, A, np);
  NED_LAUNCH_CHECK("gen_a_kernel");
  return NEDMFT_OK;
}

// ------------------------------------------------------------------ record a device failure

__device__ __forceinline__ void record_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// ------------------------------------------------------------------ in-shared-memory Gauss-Jordan

// In-place inverse of the n x n matrix `a` (row stride ld) held in shared
// memory, no pivoting (the static row order makes the pivots safe), all
// threads of the block participating.  `col` is n scratch entries.
__device__ void smem_gauss_jordan(double2* a, int n, int ld, double2* col, double tiny, int* status) {
  for (int k = 0; k < n; ++k) {
    for (int t = threadIdx.x; t < n; t += blockDim.x) col[t] = a[t * ld + k];
    __syncthreads();
    double2 pinv;
    bool ok = cinv_guard(col[k], pinv, tiny);
    if (!ok && threadIdx.x == 0) record_status(status, DS_SINGULAR);
    for (int t = threadIdx.x; t < n; t += blockDim.x) a[k * ld + t] = (t == k) ? pinv : cmul(a[k * ld + t], pinv);
    __syncthreads();
    for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
      int i = e / n, j = e % n;
      if (i == k) continue;
      double2 f = col[i];
      if (j == k) {
        double2 v = cmul(f, pinv);
        a[i * ld + k] = make_double2(-v.x, -v.y);
      } else {
        double2 v = a[i * ld + j];
        double2 r = a[k * ld + j];
        v.x -= f.x * r.x - f.y * r.y;
        v.y -= f.x * r.y + f.y * r.x;
        a[i * ld + j] = v;
      }
    }
    __syncthreads();
  }
}

// Small N_c: one CTA per point generates A'_q in shared memory, inverts it
// and writes G_q (columns un-cycled) in FP64 to out[b].
__global__ void __launch_bounds__(512) gj_small_fp64_kernel(ContourDev c, ModelDev m, const double* __restrict__ eps_d,
                                                            const double* __restrict__ ebar_d, int q0,
                                                            const double2* __restrict__ S, double2* __restrict__ out,
                                                            int* status) {
  extern __shared__ double2 sm[];
  const int n = c.n, b = blockIdx.x;
  double2* a = sm;
  double2* col = sm + n * n;
  const double eps = eps_d[q0 + b], ebar = ebar_d[q0 + b];
  const bool sh = shifted_point(m, eps);
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    int r = e / n, j = e % n;
    int i = sh ? (r + 1 == n ? 0 : r + 1) : r;
    a[e] = a_entry(c, m, eps, ebar, S, i, j);
  }
  __syncthreads();
  smem_gauss_jordan(a, n, n, col, 1e-12, status);
  double2* o = out + (size_t)b * n * n;
  for (int e = threadIdx.x; e < n * n; e += blockDim.x) {
    int i = e / n, j = e % n;
    o[e] = a[i * n + unshift_col(j, n, sh)];
  }
}

int small_path_max_n() { return kSmallPathMaxN; }

int launch_gj_small_fp64(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, int q0,
                         int nb, const double2* S, double2* out, int* status, cudaStream_t st) {
  size_t smem = (size_t)(c.n * c.n + c.n) * sizeof(double2);
  int rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj_small_fp64_kernel), 227 * 1024);
  if (rc) return rc;
  gj_small_fp64_kernel<<<nb, 512, smem, st>>>(c, m, eps, ebar, q0, S, out, status);
  NED_LAUNCH_CHECK("gj_small_fp64_kernel");
  return NEDMFT_OK;
}

// ------------------------------------------------------------------ FP64 reductions over the points

// gloc[i][j] (= or +=) sum_b wq[q0+b] X[b][i][col(j)], col = unshift_col if
// `cycled` (the batch holds X' = (P A)^-1 in boxes, box_off).  32 consecutive entries per CTA, a
// warp per eighth of the points: each sums its consecutive points in ascending
// order with eight loads in flight, then the eighths are added in order (a fixed
// order).  Bound by the loads' latency while the result is small: 135 us with a
// thread per entry over all 256 points of 80 x 80.
constexpr int kRedGroups = 8;
__global__ void __launch_bounds__(32 * kRedGroups)
    reduce_gloc_kernel(ContourDev c, ModelDev m, const double* __restrict__ eps_d, const double* __restrict__ wq_d,
                       int q0, int nb, const double2* __restrict__ X, int ldx, bool cycled, bool first,
                       double2* __restrict__ gloc) {
  __shared__ double2 part[kRedGroups][32];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const size_t total = (size_t)c.n * c.n, bstride = (size_t)ldx * ldx;
  const int b0 = (int)((long long)g * nb / kRedGroups), b1 = (int)((long long)(g + 1) * nb / kRedGroups);
  for (size_t e0 = (size_t)blockIdx.x * 32; e0 < total; e0 += (size_t)gridDim.x * 32) {  // the same trips for a CTA
    const size_t e = e0 + lane, ec = e < total ? e : 0;
    const int i = (int)(ec / c.n), j = (int)(ec - (size_t)i * c.n);
    const double2* x0 = X + (cycled ? box_off(ldx, i, j) : (size_t)i * ldx + j);
    const double2* x1 = X + (cycled ? box_off(ldx, i, unshift_col(j, c.n, true)) : 0);
    double2 acc = make_double2(0.0, 0.0);
    constexpr int U = 8;
    for (int b = b0; b < b1; b += U) {
      double2 v[U];
      double w[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int q = min(b + u, b1 - 1);
        const bool sh = cycled && shifted_point(m, eps_d[q0 + q]);
        v[u] = (sh ? x1 : x0)[(size_t)q * bstride];
        w[u] = wq_d[q0 + q];
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (b + u < b1) {
          acc.x = fma(w[u], v[u].x, acc.x);
          acc.y = fma(w[u], v[u].y, acc.y);
        }
    }
    part[g][lane] = acc;
    __syncthreads();
    if (g == 0 && e < total) {
      double2 s = first ? make_double2(0.0, 0.0) : gloc[e];
#pragma unroll
      for (int k = 0; k < kRedGroups; ++k) s = cadd(s, part[k][lane]);
      gloc[e] = s;
    }
    __syncthreads();
  }
}

// jacc[m] (= or +=) sum_b wq ebar_q(t_m) G_q[m][2 N_t - m]: a warp per time,
// lane l the points l, l + 32, ..., the lanes' sums added in a fixed tree.  The
// field's sine and cosine are the time's, not the point's (287 us with a thread
// per time and a sincos per point, 256 points).
__global__ void __launch_bounds__(128) reduce_current_kernel(ContourDev c, ModelDev mo,
                                                             const double* __restrict__ eps_d,
                                                             const double* __restrict__ ebar_d,
                                                             const double* __restrict__ wq_d, int q0, int nb,
                                                             const double2* __restrict__ X, int ldx, bool cycled,
                                                             bool first, double2* __restrict__ jacc) {
  const int mm = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (mm >= c.nt) return;  // whole warps
  const double t = t_re(c, mm);
  const int jcol = 2 * c.nt - mm;
  double sn = 0.0, cs = 1.0;  // ebar_q(t) = ebar cos(Et) + eps sin(Et), ebar before the field
  if (t > 0.0) sincos(mo.E * t, &sn, &cs);
  double2 part = make_double2(0.0, 0.0);
#pragma unroll 4
  for (int b = lane; b < nb; b += 32) {
    const int q = q0 + b;
    const double eps = eps_d[q];
    const double2 v = X[(size_t)b * ldx * ldx + (cycled ? box_off(ldx, mm, unshift_col(jcol, c.n, shifted_point(mo, eps)))
                                                        : (size_t)mm * ldx + jcol)];
    const double w = wq_d[q] * (ebar_d[q] * cs + eps * sn);
    part.x = fma(w, v.x, part.x);
    part.y = fma(w, v.y, part.y);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    part.x += __shfl_xor_sync(0xffffffffu, part.x, o);
    part.y += __shfl_xor_sync(0xffffffffu, part.y, o);
  }
  if (lane == 0) {
    const double2 acc = first ? make_double2(0.0, 0.0) : jacc[mm];
    jacc[mm] = cadd(acc, part);
  }
}

// j = Re(i acc) = -acc.y, j_imag = Im(i acc) = acc.x.
__global__ void finish_current_kernel(int nt, const double2* __restrict__ jacc, double* __restrict__ j,
                                      double* __restrict__ ji) {
  const int mm = blockIdx.x * blockDim.x + threadIdx.x;
  if (mm >= nt) return;
  if (j) j[mm] = -jacc[mm].y;
  if (ji) ji[mm] = jacc[mm].x;
}

int launch_reduce(const ContourDev& c, const ModelDev& m, const double* eps, const double* ebar, const double* wq,
                  int q0, int nb, const double2* X, int ldx, bool cycled, bool first, double2* gloc, double2* jacc,
                  cudaStream_t st) {
  const size_t total = (size_t)c.n * c.n;
  const size_t blocks = (total + 31) / 32;
  reduce_gloc_kernel<<<(int)(blocks < 152 * 32 ? blocks : 152 * 32), 32 * kRedGroups, 0, st>>>(
      c, m, eps, wq, q0, nb, X, ldx, cycled, first, gloc);
  NED_LAUNCH_CHECK("reduce_gloc_kernel");
  if (jacc) {
    reduce_current_kernel<<<ceil_div(c.nt, 4), 128, 0, st>>>(c, m, eps, ebar, wq, q0, nb, X, ldx, cycled, first, jacc);
    NED_LAUNCH_CHECK("reduce_current_kernel");
  }
  return NEDMFT_OK;
}

int launch_finish_current(int nt, const double2* jacc, double* j, double* ji, cudaStream_t st) {
  finish_current_kernel<<<ceil_div(nt, 128), 128, 0, st>>>(nt, jacc, j, ji);
  NED_LAUNCH_CHECK("finish_current_kernel");
  return NEDMFT_OK;
}

}  // namespace nedmft
