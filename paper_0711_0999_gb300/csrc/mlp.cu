// Learned warm start of the self-energy.  The impurity step gives
//   W Sigma W = -w1 D + w1 (1 - w1) D X D,  X = inv(A0 + (1 - w1) D),
// with D the point-split difference of the M matrices (one entry per row:
// d_i at (i, i-1), indices mod N, d_i = -U W_i for i >= 1, d_0 = +U W_0).  X
// is an impurity Green's function -- smooth along the contour, of order one
// for any U, with its jump at equal contour times -- while Sigma itself carries
// factors of the step sizes at the ends of the branches.  A small MLP maps
// (U, E, dt, t, t') to X(t, t'); the self-energy follows from the identity
// above.  Forward and backward (mean-squared error) run on the tensor cores,
// all layers in one kernel (mlp_umma.cu: operands rounded to bf16, FP32 sums in
// TMEM); weights and optimizer state are FP32.
#include <math.h>

#include "common.cuh"
#include "mlp_umma.cuh"

namespace nedmft {
namespace {

constexpr int kIn = kMlpIn;    // features per (t, t') pair
constexpr int kOut = kMlpOut;  // Re, Im of the smooth Sigma part
constexpr size_t kParams = mlp_w_off(kMlpLayers);

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m1,
                            float* __restrict__ m2, size_t n, float lr, float b1, float b2, float eps, float c1,
                            float c2) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n; e += (size_t)gridDim.x * blockDim.x) {
    const float gg = g[e];
    const float a = b1 * m1[e] + (1.f - b1) * gg;
    const float b = b2 * m2[e] + (1.f - b2) * gg * gg;
    m1[e] = a;
    m2[e] = b;
    p[e] -= lr * (a / c1) / (sqrtf(b / c2) + eps);
  }
}

// Features of the pair (t_a, t_b) of X, built to carry over to contours
// longer than the training runs' (the field is switched on at t = 0; after a
// few units of time a metal's Green's function depends on t - t' alone):
// U/2.5, E/4, tanh(Re(t_a - t_b)/3), then for each time t (real part r,
// imaginary-branch depth tau) tanh(max(r, 0)/3) (the elapsed field time,
// saturating), min(r, 0)/5 (the time before the field), tau/beta and the
// branch one-hot (upper, lower, imaginary), then the contour order
// theta_c(t_a, t_b) (1 for a >= b), across which X jumps, and dt / 0.1 (the
// discrete X differs from the continuum one at order dt, so the network learns
// it at the training steps and the warm start extrapolates in dt).
__device__ __forceinline__ void row_features(const ContourDev& c, int k, float* f) {
  const double r = t_re(c, k);
  f[0] = (float)tanh(fmax(r, 0.0) / 3.0);
  f[1] = (float)(fmin(r, 0.0) / 5.0);
  f[2] = (float)(t_tau(c, k) / c.beta);
  f[3] = k < c.nt ? 1.f : 0.f;
  f[4] = (k >= c.nt && k < 2 * c.nt) ? 1.f : 0.f;
  f[5] = k >= 2 * c.nt ? 1.f : 0.f;
}
__global__ void features_kernel(ContourDev c, ModelDev m, double dt_feature, float* __restrict__ x) {
  const size_t total = (size_t)c.n * c.n;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int i = (int)(e / c.n), j = (int)(e % c.n);
    float* f = x + e * kIn;
    f[0] = (float)(m.U / 2.5);
    f[1] = (float)(m.E / 4.0);
    f[2] = (float)tanh((t_re(c, i) - t_re(c, j)) / 3.0);
    row_features(c, i, f + 3);
    row_features(c, j, f + 9);
    f[15] = i >= j ? 1.f : 0.f;
    f[16] = (float)(dt_feature / 0.1);
  }
}
// The same for the warm start, which needs them once for all its training steps
// and never as 17 floats per pair in memory: six values per row, and the tanh of
// the relative time, an odd function, for the pairs a <= b, written to both
// places (FP64 tanh is what this kernel is bound by: 1.7 ms for two steps of
// N_c = 1500 when every pair of every step evaluated three).
__global__ void __launch_bounds__(256) pair_features_kernel(ContourDev c, float* __restrict__ row,
                                                            float* __restrict__ rel) {
  const int i = blockIdx.x;
  if (threadIdx.x == 0) row_features(c, i, row + (size_t)i * 6);
  for (int j = i + threadIdx.x; j < c.n; j += blockDim.x) {
    const float v = (float)tanh((t_re(c, i) - t_re(c, j)) / 3.0);
    rel[(size_t)i * c.n + j] = v;
    if (j != i) rel[(size_t)j * c.n + i] = -v;
  }
}

// d_i, the entry of D in row i (column i - 1 mod N).
__device__ __forceinline__ double2 d_entry(const ContourDev& c, double U, int i) {
  const double2 w = weight(c, i);
  return i == 0 ? make_double2(U * w.x, U * w.y) : make_double2(-U * w.x, -U * w.y);
}

// Sigma from X: W Sigma W = -w1 D + w1 (1 - w1) D X D, i.e.
// Sigma_ij = [-w1 D_ij + w1 (1 - w1) d_i X[i-1][j+1] d_{j+1}] / (W_i W_j)
// (indices mod N); X[a][b] is the complex value y[(a N + b)] (Re, Im).  A row
// per CTA: the factors of X that depend on i or j alone, d_i / W_i and d_{j+1} /
// W_j, are formed once per row and once per column chunk, so an entry costs two
// complex products (251 us at N_c = 1500 when every entry formed and divided by
// W_i W_j in FP64).
__global__ void __launch_bounds__(256) assemble_sigma_kernel(ContourDev c, ModelDev m, const float* __restrict__ y,
                                                             double2* __restrict__ sigma) {
  constexpr int kRowsPer = 16;
  const int n = c.n, i0 = blockIdx.y * kRowsPer;
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  auto over = [](double2 a, double2 w) {
    const double m2 = w.x * w.x + w.y * w.y;
    return cmul(a, make_double2(w.x / m2, -w.y / m2));
  };
  const double w1 = m.w1;
  const int jn = j + 1 >= n ? 0 : j + 1;
  const double2 wj = weight(c, j < n ? j : 0);
  double2 fj = over(d_entry(c, m.U, jn), wj);
  fj = make_double2(w1 * (1.0 - w1) * fj.x, w1 * (1.0 - w1) * fj.y);
  __shared__ double2 fi[kRowsPer];
  if (threadIdx.x < kRowsPer && i0 + threadIdx.x < n)
    fi[threadIdx.x] = over(d_entry(c, m.U, i0 + threadIdx.x), weight(c, i0 + threadIdx.x));
  __syncthreads();
  if (j >= n) return;
  for (int r = 0; r < kRowsPer && i0 + r < n; ++r) {
    const int i = i0 + r, ip = i == 0 ? n - 1 : i - 1;
    const size_t f = (size_t)ip * n + jn;
    double2 v = cmul(cmul(fi[r], make_double2(y[2 * f], y[2 * f + 1])), fj);
    if (j == ip) {  // - w1 d_i / (W_i W_j)
      const double2 d = over(fi[r], wj);
      v = make_double2(v.x - w1 * d.x, v.y - w1 * d.y);
    }
    sigma[(size_t)i * n + j] = v;
  }
}

// The training target X[a][b] = [W Sigma W + w1 D]_{a+1, b-1} / (w1 (1 - w1) d_{a+1} d_b), / scale.
__global__ void target_kernel(ContourDev c, ModelDev m, const double2* __restrict__ sigma, double inv_scale,
                              float* __restrict__ t) {
  const int n = c.n;
  const size_t total = (size_t)n * n;
  const double w1 = m.w1;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int a = (int)(e / n), b = (int)(e % n);
    const int i = a + 1 == n ? 0 : a + 1, j = b == 0 ? n - 1 : b - 1;
    const double2 di = d_entry(c, m.U, i);
    double2 v = cmul(cmul(weight(c, i), sigma[(size_t)i * n + j]), weight(c, j));
    if (j == (i == 0 ? n - 1 : i - 1)) v = make_double2(v.x + w1 * di.x, v.y + w1 * di.y);
    const double2 den = cmul(di, d_entry(c, m.U, b));
    const double dm = w1 * (1.0 - w1) * (den.x * den.x + den.y * den.y);
    v = cmul(v, make_double2(den.x / dm, -den.y / dm));
    t[2 * e] = (float)(v.x * inv_scale);
    t[2 * e + 1] = (float)(v.y * inv_scale);
  }
}

int grid_for(size_t n) {
  size_t b = (n + 255) / 256;
  return (int)(b > 152 * 16 ? 152 * 16 : (b < 1 ? 1 : b));
}

}  // namespace
}  // namespace nedmft

using namespace nedmft;

extern "C" int32_t nedmft_mlp_param_count(void) { return (int32_t)kParams; }

extern "C" size_t nedmft_mlp_workspace_size(int32_t n) {
  if (n < 1) return 0;
  return mlp_grad_scratch(n) + 256;  // the scratch is aligned to 256 bytes inside
}

extern "C" int nedmft_mlp_forward(const float* params_d, const float* x_d, int32_t n, float* y_d, void* ws_d,
                                  size_t ws_bytes, void* stream) {
  if (!params_d || !x_d || !y_d || !ws_d || n < 1) return set_error(NEDMFT_EINVAL, "mlp_forward: bad argument");
  if (ws_bytes < nedmft_mlp_workspace_size(n)) return set_error(NEDMFT_ENOMEM, "mlp_forward: workspace too small");
  MlpInput in;
  in.x = x_d;
  return mlp_forward(params_d, in, n, y_d, false, true, 1.f, true, align256(ws_d),
                     static_cast<cudaStream_t>(stream));
}

extern "C" int nedmft_mlp_grad(const float* params_d, const float* x_d, const float* target_d, int32_t n,
                               float* grad_d, float* loss_d, void* ws_d, size_t ws_bytes, void* stream) {
  if (!params_d || !x_d || !target_d || !grad_d || !loss_d || !ws_d || n < 1)
    return set_error(NEDMFT_EINVAL, "mlp_grad: bad argument");
  if (ws_bytes < nedmft_mlp_workspace_size(n)) return set_error(NEDMFT_ENOMEM, "mlp_grad: workspace too small");
  return mlp_gradient(params_d, x_d, target_d, n, grad_d, loss_d, align256(ws_d),
                      static_cast<cudaStream_t>(stream));
}

extern "C" int nedmft_mlp_adam(float* params_d, const float* grad_d, float* m1_d, float* m2_d, int32_t step, float lr,
                               void* stream) {
  if (!params_d || !grad_d || !m1_d || !m2_d || step < 1) return set_error(NEDMFT_EINVAL, "mlp_adam: bad argument");
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)step), c2 = 1.f - powf(b2, (float)step);
  adam_kernel<<<grid_for(kParams), 256, 0, static_cast<cudaStream_t>(stream)>>>(params_d, grad_d, m1_d, m2_d, kParams,
                                                                                 lr, b1, b2, 1e-8f, c1, c2);
  NED_LAUNCH_CHECK("adam_kernel");
  return NEDMFT_OK;
}

extern "C" int nedmft_mlp_features(const nedmft_contour* c, const nedmft_model* m, float* x_d, void* stream) {
  if (!c || !m || !x_d || c->n_c < 1) return set_error(NEDMFT_EINVAL, "mlp_features: bad argument");
  const ContourDev cd = to_dev(*c);
  const ModelDev md{m->U, m->E, m->w1, isnan(m->mu) ? m->U / 2 : m->mu};
  features_kernel<<<grid_for((size_t)cd.n * cd.n), 256, 0, static_cast<cudaStream_t>(stream)>>>(cd, md, cd.dt, x_d);
  NED_LAUNCH_CHECK("features_kernel");
  return NEDMFT_OK;
}

extern "C" int nedmft_mlp_target(const nedmft_contour* c, const nedmft_model* m, const nedmft_c128* sigma_d,
                                 double scale, float* t_d, void* stream) {
  if (!c || !m || !sigma_d || !t_d || !(scale > 0)) return set_error(NEDMFT_EINVAL, "mlp_target: bad argument");
  const ContourDev cd = to_dev(*c);
  const ModelDev md{m->U, m->E, m->w1, isnan(m->mu) ? m->U / 2 : m->mu};
  target_kernel<<<grid_for((size_t)cd.n * cd.n), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      cd, md, reinterpret_cast<const double2*>(sigma_d), 1.0 / scale, t_d);
  NED_LAUNCH_CHECK("target_kernel");
  return NEDMFT_OK;
}

extern "C" size_t nedmft_sigma_warm_start_workspace_size(const nedmft_contour* c) {
  if (!c || c->n_c < 1) return 0;
  const size_t n = c->n_c;
  return mlp_forward_scratch() + align256(sizeof(float) * n * 6) + align256(sizeof(float) * n * n) +
         align256(sizeof(float) * n * n * kOut) + 256;
}

extern "C" int nedmft_sigma_warm_start(const nedmft_contour* c, const nedmft_model* m, const float* params_d,
                                       int32_t n_dt, const double* dts_host, nedmft_c128* sigma_d, void* ws_d,
                                       size_t ws_bytes, void* stream) {
  if (!c || !m || !params_d || !sigma_d || !ws_d || !dts_host || n_dt < 1 || n_dt > 8)
    return set_error(NEDMFT_EINVAL, "sigma_warm_start: bad argument");
  if (!(m->U != 0.0) || !(m->w1 > 0.0 && m->w1 < 1.0))
    return set_error(NEDMFT_EINVAL, "sigma_warm_start: needs U != 0 and 0 < w1 < 1");
  for (int k = 0; k < n_dt; ++k)
    for (int q = 0; q < k; ++q)
      if (!(dts_host[k] > 0.0) || dts_host[k] == dts_host[q])
        return set_error(NEDMFT_EINVAL, "sigma_warm_start: steps must be positive and distinct");
  if (ws_bytes < nedmft_sigma_warm_start_workspace_size(c))
    return set_error(NEDMFT_ENOMEM, "sigma_warm_start: workspace too small");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const size_t n = c->n_c, n2 = n * n;
  char* p = align256(ws_d);
  char* scratch = p; p += mlp_forward_scratch();
  float* row = reinterpret_cast<float*>(p); p += align256(sizeof(float) * n * 6);
  float* rel = reinterpret_cast<float*>(p); p += align256(sizeof(float) * n2);
  float* y = reinterpret_cast<float*>(p);
  const ContourDev cd = to_dev(*c);
  const ModelDev md{m->U, m->E, m->w1, isnan(m->mu) ? m->U / 2 : m->mu};
  pair_features_kernel<<<(int)n, 256, 0, st>>>(cd, row, rel);
  NED_LAUNCH_CHECK("pair_features_kernel");
  MlpInput in;
  in.row = row;
  in.rel = rel;
  in.nc = (int)n;
  in.u = (float)(md.U / 2.5);
  in.e = (float)(md.E / 4.0);
  for (int k = 0; k < n_dt; ++k) {
    // X at the step dts[k] on this contour's times, weighted by the Lagrange
    // basis polynomial of dts[k] at this contour's step (extrapolation in dt)
    double lk = 1.0;
    for (int q = 0; q < n_dt; ++q)
      if (q != k) lk *= (cd.dt - dts_host[q]) / (dts_host[k] - dts_host[q]);
    in.dt = (float)(dts_host[k] / 0.1);
    if (int rc = mlp_forward(params_d, in, n2, y, true, k == 0, (float)lk, k == 0, scratch, st)) return rc;
  }
  assemble_sigma_kernel<<<dim3(ceil_div((int)n, 256), ceil_div((int)n, 16)), 256, 0, st>>>(
      cd, md, y, reinterpret_cast<double2*>(sigma_d));
  NED_LAUNCH_CHECK("assemble_sigma_kernel");
  return NEDMFT_OK;
}

namespace nedmft {
namespace {
// x_b[r] = x[idx(r)], t_b[r] = t[idx(r)], idx from a counter-based hash of
// (seed, step, r) (splitmix64 finaliser) modulo n_total.
__global__ void sample_kernel(const float* __restrict__ x, const float* __restrict__ t, long long n_total, int batch,
                              unsigned long long seed, long long step, float* __restrict__ xb, float* __restrict__ tb) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= batch) return;
  unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(step * (long long)batch + r + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z ^= z >> 31;
  const long long i = (long long)(z % (unsigned long long)n_total);
  for (int f = 0; f < kIn; ++f) xb[(size_t)r * kIn + f] = x[(size_t)i * kIn + f];
  for (int f = 0; f < kOut; ++f) tb[(size_t)r * kOut + f] = t[(size_t)i * kOut + f];
}
}  // namespace
}  // namespace nedmft

extern "C" int nedmft_mlp_sample(const float* x_d, const float* t_d, int64_t n_total, int32_t batch, uint64_t seed,
                                 int64_t step, float* xb_d, float* tb_d, void* stream) {
  if (!x_d || !t_d || !xb_d || !tb_d || n_total < 1 || batch < 1)
    return set_error(NEDMFT_EINVAL, "mlp_sample: bad argument");
  sample_kernel<<<ceil_div(batch, 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(x_d, t_d, n_total, batch, seed,
                                                                                      step, xb_d, tb_d);
  NED_LAUNCH_CHECK("sample_kernel");
  return NEDMFT_OK;
}
