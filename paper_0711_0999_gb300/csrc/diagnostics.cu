// Accuracy diagnostics of a converged contour Green's function (Sec. II): the
// equal-time moments of the retarded function and the nonequilibrium density
// of states of Eqs. gr_omega and dos_def.  FP64 throughout.
#include <math.h>

#include "lattice.cuh"

namespace nedmft {
namespace {

// G^R(t_i, t_j) = G^>(t_i, t_j) - G^<(t_i, t_j) on the real branches, i >= j:
// G^> is the element (lower-branch row of t_i, upper row of t_j), G^< the
// element (upper row of t_i, lower row of t_j); the lower-branch row of t_m
// is 2 N_t - m (for t_min the first imaginary point).
__device__ __forceinline__ double2 retarded_at(const double2* __restrict__ g, int n, int nt, int i, int j) {
  const double2 gt = g[(size_t)(2 * nt - i) * n + j];
  const double2 lt = g[(size_t)i * n + (2 * nt - j)];
  return make_double2(gt.x - lt.x, gt.y - lt.y);
}

// f(s) = i G^R(t_m + s/2, t_m - s/2) = mu0 - i mu1 s - mu2 s^2 / 2 + ...: the
// quadratic through s = h, 2h, 3h (h = 2 dt) has value 3 f1 - 3 f2 + f3 at 0,
// slope (-5 f1 + 8 f2 - 3 f3) / 2h and curvature (f1 - 2 f2 + f3) / 2h^2.
__global__ void moments_kernel(const double2* __restrict__ g, int n, int nt, double dt, double* __restrict__ mu0,
                               double* __restrict__ mu1, double* __restrict__ mu2, double* __restrict__ dens) {
  const int m = blockIdx.x * blockDim.x + threadIdx.x;
  if (m >= nt) return;
  if (dens) dens[m] = g[(size_t)m * n + (2 * nt - m)].y;  // n = -i G^< with G^< = i n
  double a0 = NAN, a1 = NAN, a2 = NAN;
  if (m >= 3 && m + 3 < nt) {
    double2 f[3];
#pragma unroll
    for (int k = 1; k <= 3; ++k) {
      const double2 r = retarded_at(g, n, nt, m + k, m - k);
      f[k - 1] = make_double2(-r.y, r.x);  // i G^R
    }
    const double h = 2.0 * dt;
    const double2 v0 = make_double2(3.0 * f[0].x - 3.0 * f[1].x + f[2].x, 3.0 * f[0].y - 3.0 * f[1].y + f[2].y);
    const double2 v1 = make_double2((-5.0 * f[0].x + 8.0 * f[1].x - 3.0 * f[2].x) / (2.0 * h),
                                    (-5.0 * f[0].y + 8.0 * f[1].y - 3.0 * f[2].y) / (2.0 * h));
    const double2 v2 = make_double2((f[0].x - 2.0 * f[1].x + f[2].x) / (2.0 * h * h),
                                    (f[0].y - 2.0 * f[1].y + f[2].y) / (2.0 * h * h));
    a0 = v0.x;
    a1 = -v1.y;  // Re(i v1)
    a2 = -2.0 * v2.x;
  }
  if (mu0) mu0[m] = a0;
  if (mu1) mu1[m] = a1;
  if (mu2) mu2[m] = a2;
}

// rho(t_m, omega) = -Im G^R(t_m, omega) / pi with the trapezoid rule over the
// relative times 2 k dt, k = 0 .. min(m, N_t - 1 - m).  Block x: average time
// m_list[x]; a warp per omega.  The weighted G^R of up to 1024 relative times is
// staged once per CTA; lane l sums the B consecutive terms from l B on with the
// phases e^{i omega b h}, b < B, which lane b has formed for the whole warp, and
// multiplies its sum by e^{i omega l B h}: two sincos per lane for up to 1024
// terms where a thread per omega formed one per term (455 us for 5 times x 401
// frequencies of N_c = 1500 on 20 CTAs, serial in k).  What is left is latency:
// the staging loads and one sincos after another.
// With few relative times those 64 sincos of a frequency are more than its terms:
// up to `direct` times, a lane per omega, the terms dealt to the CTA's warps.
// FP64 bound: K sincos per frequency.  The line: 64 terms where 32 frequencies per
// SM keep all of them busy, else 16, the eight warps' sincos of the other form on
// one SM (up to 10 relative times, 5 averages x 100000 and 12 x 1000 frequencies:
// 2455 and 91 us with a warp per omega, 244 and 43 so).
// CTAs along y take frequencies in strides.
constexpr int kDosTerms = 1024;
constexpr int kDosWarps = 8;
__global__ void __launch_bounds__(32 * kDosWarps)
    dos_kernel(const double2* __restrict__ g, int n, int nt, double dt, const int* __restrict__ m_list,
               const double* __restrict__ omega, int n_omega, int direct, double* __restrict__ rho) {
  __shared__ double2 term[kDosTerms];
  __shared__ double part[kDosWarps][32];
  const int a = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = m_list[a];
  const bool inside = m >= 0 && m < nt;
  const int kmax = inside ? min(m, nt - 1 - m) : 0;  // the same for the whole CTA
  const double h = 2.0 * dt;
  auto stage = [&](int k0, int cnt) {
    for (int k = threadIdx.x; k < cnt; k += blockDim.x) {
      const double2 r = retarded_at(g, n, nt, m + k0 + k, m - k0 - k);
      const double wk = (k0 + k == 0 || k0 + k == kmax) ? 0.5 * h : h;
      term[k] = make_double2(wk * r.x, wk * r.y);
    }
  };
  auto store = [&](unsigned w, double im) {
    rho[(size_t)a * n_omega + w] = !inside ? NAN : kmax == 0 ? 0.0 : -im / M_PI;
  };
  if (kmax < direct) {
    if (blockIdx.y * 32u >= (unsigned)n_omega) return;
    if (kmax > 0) stage(0, kmax + 1);
    __syncthreads();
    for (unsigned w0 = blockIdx.y * 32u; w0 < (unsigned)n_omega; w0 += gridDim.y * 32u) {
      const unsigned w = w0 + lane;
      const double om = w < (unsigned)n_omega ? omega[w] : 0.0;
      double im = 0.0;
      for (int k = warp; kmax > 0 && k <= kmax; k += kDosWarps) {
        double sn, cs;
        sincos(om * (k * h), &sn, &cs);
        im += cs * term[k].y + sn * term[k].x;  // Im(e^{i om s} G^R)
      }
      part[warp][lane] = im;
      __syncthreads();
      if (warp == 0 && w < (unsigned)n_omega) {
        for (int q = 1; q < kDosWarps; ++q) im += part[q][lane];
        store(w, im);
      }
      __syncthreads();
    }
    return;
  }
  for (unsigned w0 = blockIdx.y * kDosWarps; w0 < (unsigned)n_omega; w0 += gridDim.y * kDosWarps) {
    const unsigned w = w0 + warp;
    const double om = w < (unsigned)n_omega ? omega[w] : 0.0;
    double im = 0.0;
    for (int k0 = 0; k0 <= kmax; k0 += kDosTerms) {
      const int cnt = min(kDosTerms, kmax + 1 - k0);
      const int B = ((cnt + 31) >> 5) | 1;  // odd: the lanes' terms fall on different banks
      __syncthreads();
      stage(k0, cnt);
      __syncthreads();
      double bs, bc, ls, lc;
      sincos(om * (lane * h), &bs, &bc);
      double2 p = make_double2(0.0, 0.0);
      const int l0 = lane * B;
      for (int b0 = 0; b0 < B; b0 += 32) {  // B is 33 when 1024 terms are staged
        if (b0 > 0) sincos(om * ((b0 + lane) * h), &bs, &bc);
        const int nb = min(32, B - b0);
        for (int b = 0; b < nb; ++b) {
          const double c = __shfl_sync(0xffffffffu, bc, b), sn = __shfl_sync(0xffffffffu, bs, b);
          if (l0 + b0 + b < cnt) {
            const double2 r = term[l0 + b0 + b];
            p.x = fma(c, r.x, fma(-sn, r.y, p.x));
            p.y = fma(c, r.y, fma(sn, r.x, p.y));
          }
        }
      }
      if (l0 < cnt) {
        // one phase for B terms: the rounding of its angle, which they would share, is put back
        const double k = (double)(k0 + l0), t = k * h, te = fma(k, h, -t);
        const double an = om * t;
        double ae = fma(om, t, -an) + om * te;
        if (fabs(ae) > 0x1p-26) ae = 0.0;  // |om t| beyond 2^27: no more than a lone term's angle has
        sincos(an, &ls, &lc);
        const double s1 = fma(lc, ae, ls), c1 = fma(-ls, ae, lc);
        im += c1 * p.y + s1 * p.x;  // Im(e^{i om s} G^R)
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) im += __shfl_xor_sync(0xffffffffu, im, o);
    if (lane == 0 && w < (unsigned)n_omega) store(w, im);
  }
}

}  // namespace
}  // namespace nedmft

using namespace nedmft;

extern "C" int nedmft_moments(const nedmft_contour* c, const nedmft_c128* gloc_d, double* mu0_d, double* mu1_d,
                              double* mu2_d, double* dens_d, void* stream) {
  if (!c || !gloc_d) return set_error(NEDMFT_EINVAL, "moments: NULL argument");
  if (c->n_t < 1 || c->n_tau < 1 || c->n_c != 2 * c->n_t + c->n_tau || !(c->dt > 0))
    return set_error(NEDMFT_EINVAL, "moments: invalid contour");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  moments_kernel<<<ceil_div(c->n_t, 128), 128, 0, st>>>(reinterpret_cast<const double2*>(gloc_d), c->n_c, c->n_t,
                                                        c->dt, mu0_d, mu1_d, mu2_d, dens_d);
  NED_LAUNCH_CHECK("moments_kernel");
  return NEDMFT_OK;
}

extern "C" int nedmft_dos(const nedmft_contour* c, const nedmft_c128* gloc_d, const int32_t* m_d, int32_t n_avg,
                          const double* omega_d, int32_t n_omega, double* rho_d, void* stream) {
  if (!c || !gloc_d) return set_error(NEDMFT_EINVAL, "dos: NULL argument");
  if (c->n_t < 1 || c->n_tau < 1 || c->n_c != 2 * c->n_t + c->n_tau || !(c->dt > 0))
    return set_error(NEDMFT_EINVAL, "dos: invalid contour");
  if (n_avg < 0 || n_omega < 0 || n_avg > 65535) return set_error(NEDMFT_EINVAL, "dos: bad sizes");
  if (n_avg == 0 || n_omega == 0) return NEDMFT_OK;  // nothing to write; the arrays may be NULL
  if (!m_d || !omega_d || !rho_d) return set_error(NEDMFT_EINVAL, "dos: NULL argument");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  constexpr long long kSms = 152;
  const long long total = (long long)n_avg * n_omega;
  const int direct = total >= 32 * kSms ? 64 : 16;
  // 32 frequencies per CTA where that leaves 32 CTAs per SM (fewer idle CTAs with few relative times); at most
  // 65535 CTAs along y, which take every so many frequencies past that
  const int per = total >= 1024 * kSms ? 32 : kDosWarps;
  const int blocks = (int)(((long long)n_omega + per - 1) / per);
  dos_kernel<<<dim3(n_avg, blocks < 65535 ? blocks : 65535), 32 * kDosWarps, 0, st>>>(
      reinterpret_cast<const double2*>(gloc_d), c->n_c, c->n_t, c->dt, m_d, omega_d, n_omega, direct, rho_d);
  NED_LAUNCH_CHECK("dos_kernel");
  return NEDMFT_OK;
}
