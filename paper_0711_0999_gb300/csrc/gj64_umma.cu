// Batched FP64 Gauss-Jordan inversion on the tensor cores (the FP64 lattice
// path):  step K (32 columns) of every np x np matrix is
//   P = inv(A_KK)                                   gj64_pivot_kernel
//   C = A_{:,K} with C_K = -I, cut into digits      gj64_pivot_kernel (its other CTAs)
//   R = P A_{K,:} with R_K = P, cut into digits     gj64_rpanel_kernel
//   A <- A (rows and columns K zeroed) - C R        gj64_update_kernel
// No pivoting: the caller's row order makes every multiplier at most one.
//
// Why the tensor cores: GB300 has two FP64 FMA units per SM (1.26 TFLOP/s),
// so the 8 n^3 operations of an inverse bound the CUDA-core form it replaces
// (20.6 ms per matrix at n = 1500).  Here every product runs as an Ozaki split:
// a row of C (or a column of R, of P, of A_K) is scaled by a power of two to
// below one and cut into kS = 7 balanced base-256 digits, X = round(x 2^(55-e))
// = sum_s q_s 256^(6-s), |q_s| <= 128, exact in bf16.  A digit product summed
// over the 64 reals of K is below 2^20 and the up to seven products of one
// order o = a + b below 7 2^20 < 2^24, so FP32 accumulation in TMEM is exact.
// The 28 products of order <= 6 are kept (what is left out is 2^-56 of the row
// and column maxima), their sums are put together in 64-bit integers and
// rounded once to FP64: the result carries less rounding than 64 FP64 FMAs.
//
// One MMA per digit a of the left operand takes all its partners b = 0 .. 6-a
// at once: the right operand's digits lie back to back in shared memory, and
// orders a .. 6 back to back in TMEM.
#include "lattice.cuh"
#include "umma_core.cuh"

namespace nedmft {

using namespace umma;

namespace {

constexpr int kS = 7;    // digits of an operand, orders kept
constexpr int kNB = 32;  // complex columns per step
constexpr int kK = 64;   // reals per row of C and column of R: [re | im]
constexpr int kTn = 16;  // complex columns of an update tile
constexpr int kARow = kTileElems;            // bf16 elements of one digit of a 128-row tile
constexpr int kATile = kS * kTileElems;      // ... of all digits
constexpr int kBDig = 2 * kTn * kK;          // bf16 elements of one digit of a 16-column tile of R
constexpr int kBTile = kS * kBDig;

// ------------------------------------------------------------------ digits

// |x| as ordered bits of its upper word: a maximum over these gives the
// exponent of the largest value without an FP64 instruction.
__device__ __forceinline__ unsigned mag_hi(double v) { return (unsigned)__double2hiint(v) & 0x7fffffffu; }

// Biased exponent a row is scaled by, from the largest mag_hi of its values.
// Rows below 2^-450 are scaled as if at 2^-450 (their digits vanish with them).
__device__ __forceinline__ int row_biased(unsigned m) { return max((int)(m >> 20), 1023 - 450); }

// Y = X + 0x808080808080 with X = round(v 2^(55-e)), e = be - 1022: byte b <
// 6 of Y less 128 is digit 6 - b of v, Y >> 48 (signed) digit 0.  Integer
// instructions only (the FP64 units have work of their own).
__device__ __forceinline__ long long digit_word(double v, int be) {
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
  const int ex = (int)((hi >> 20) & 0x7ff);
  const int sr = be - ex;  // >= 0
  unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 2;
  m = (sr > 56 || ex == 0) ? 0 : (m + ((1ull << sr) >> 1)) >> sr;
  const long long x = (int)hi < 0 ? -(long long)m : (long long)m;
  return x + 0x808080808080ll;
}
// digit s of two values as a pair of bf16
template <int S>
__device__ __forceinline__ uint32_t digit_pair(long long y0, long long y1) {
  float f0, f1;
  if constexpr (S == 0) {  // signed, |q| <= 128: 1.5 2^23 + q less 1.5 2^23
    f0 = __int_as_float(0x4B400000 + (int)(y0 >> 48)) - 12582912.f;
    f1 = __int_as_float(0x4B400000 + (int)(y1 >> 48)) - 12582912.f;
  } else {
    constexpr int b = 6 - S;
    const uint32_t w0 = b < 4 ? (uint32_t)y0 : (uint32_t)((unsigned long long)y0 >> 32);
    const uint32_t w1 = b < 4 ? (uint32_t)y1 : (uint32_t)((unsigned long long)y1 >> 32);
    f0 = __uint_as_float(__byte_perm(w0, 0x4B000000u, 0x7440u | (b & 3))) - 8388736.f;  // 2^23 + byte, less 2^23 + 128
    f1 = __uint_as_float(__byte_perm(w1, 0x4B000000u, 0x7440u | (b & 3))) - 8388736.f;
  }
  return __byte_perm(__float_as_uint(f0), __float_as_uint(f1), 0x7632);  // exact in bf16: the upper halves
}
// the seven digits of eight values as core-matrix rows of 16 bytes: put(s, 16 bytes)
template <int S = 0, class Put>
__device__ __forceinline__ void put_digits(const long long (&y)[8], Put&& put) {
  put(S, make_uint4(digit_pair<S>(y[0], y[1]), digit_pair<S>(y[2], y[3]), digit_pair<S>(y[4], y[5]),
                    digit_pair<S>(y[6], y[7])));
  if constexpr (S + 1 < kS) put_digits<S + 1>(y, put);
}
__device__ __forceinline__ uint4 neg_bf16(uint4 v) {
  return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}
// element offset of (row, k) in a canonical K-major tile of 64 k
__device__ __forceinline__ int core_off(int row, int k) { return ((row >> 3) * 8 + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7); }

// ------------------------------------------------------------------ order sums to FP64

// 2^(e-53) sum_o c_o 2^(8(5-o)) / 2 as a double, rounded once; c_o, o = 0 .. 6,
// are integers with |c_o| <= (o + 1) 2^20.  ebase = 1023 + e - 53.
// Float to int by the 1.5 2^23 trick (below 2^22; conversion instructions run
// at an eighth of the rate), orders 4 .. 6 with the half of order 4 split off
// first; the sum as a 64-bit integer in units of 2; its leading bit found by
// the one int-to-float conversion, then shifted, rounded and assembled on the
// integer units.
__device__ __forceinline__ double orders_to_double(float c0, float c1, float c2, float c3, float c4, float c5,
                                                   float c6, int ebase) {
  constexpr float kM = 12582912.f;
  constexpr uint32_t kOff = 0x4B400000u * 257u;
  const uint32_t b0 = __float_as_uint(c0 + kM), b1 = __float_as_uint(c1 + kM);
  const uint32_t b2 = __float_as_uint(c2 + kM), b3 = __float_as_uint(c3 + kM);
  const float t4 = fmaf(c4, 0.5f, kM);
  const float rem = fmaf(c4, 0.5f, kM - t4);
  const float g = fmaf(rem, 512.f, fmaf(c6, 0.00390625f, c5));
  const uint32_t b4 = __float_as_uint(t4), b5 = __float_as_uint(fmaf(g, 0.5f, kM));
  const int u0 = (int)(b0 * 256u + b1 - kOff);
  const int u1 = (int)(b2 * 256u + b3 - kOff);
  const int u2 = (int)(b4 * 256u + b5 - kOff);
  const long long T = ((long long)u0 << 31) + (long long)u1 * 32768ll + (long long)u2;
  const unsigned long long a = T < 0 ? 0ull - (unsigned long long)T : (unsigned long long)T;
  uint32_t hi = (uint32_t)(a >> 32), lo = (uint32_t)a;
  const bool low = hi == 0;
  if (low) { hi = lo; lo = 0; }
  const uint32_t f = __float_as_uint(__uint2float_rz(hi));  // exponent 127 + index of the leading bit
  const int n = 158 - (int)(f >> 23);                       // shift that brings it to bit 31
  const uint32_t mh = __funnelshift_l(lo, hi, n), ml = lo << (n & 31);
  uint32_t ql = __funnelshift_r(ml, mh, 11), qh = mh >> 11;
  const uint32_t rnd = (ml >> 10) & 1u;
  ql += rnd;
  qh += (rnd && ql == 0) ? 1u : 0u;
  int ex = (int)(f >> 23) - 127 + (low ? 0 : 32) + ebase;  // biased exponent of the result
  ex = min(ex, 2047);                                      // beyond FP64: infinite or NaN, caught at the next digit cut
  const uint32_t rh = (qh + ((uint32_t)(ex - 1) << 20)) | (T < 0 ? 0x80000000u : 0u);
  return hi == 0 ? 0.0 : __hiloint2double((int)rh, (int)ql);
}

// ------------------------------------------------------------------ pivot block and C digits

// CTAs 0 .. nb-1: P = inv(A_KK) of matrix b, 32 x 32 FP64, a warp per four
// rows, lane = column.  Step k: the pivot row, divided by its pivot (its own
// entry replaced by the pivot's inverse), goes to shared memory (two buffers,
// one barrier per step); every other row subtracts its entry of column k times
// it, that entry counted as zero before.  FP64 bound: 32 rows x 4 FMAs x 16
// cycles per step.
// CTAs nb ..: digits of 128 rows of C, two threads per row; this work hides
// behind the pivot blocks' latency.
__global__ void __launch_bounds__(256) gj64_pivot_kernel(const double2* __restrict__ A, int np, int mtiles, int k0,
                                                         int nb, double2* __restrict__ Pbuf,
                                                         __nv_bfloat16* __restrict__ cimg, int* __restrict__ cexp,
                                                         int* status) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  if ((int)blockIdx.x < nb) {
    __shared__ double2 rowb[2][32];
    const int b = blockIdx.x;
    const double2* a = A + (size_t)b * np * np + (size_t)k0 * np + k0;
    double2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = a[(size_t)(4 * warp + q) * np + lane];
    for (int kw = 0; kw < 8; ++kw)
#pragma unroll
      for (int kq = 0; kq < 4; ++kq) {
        const int k = 4 * kw + kq, buf = k & 1;
        if (warp == kw) {
          const double2 d = make_double2(__shfl_sync(0xffffffffu, v[kq].x, k), __shfl_sync(0xffffffffu, v[kq].y, k));
          double2 pinv;
          if (!cinv_guard<double>(d, pinv, 1e-12) && lane == 0 && status) atomicCAS(status, 0, DS_SINGULAR);
          v[kq] = lane == k ? pinv : cmul(v[kq], pinv);
          rowb[buf][lane] = v[kq];
        }
        __syncthreads();
        const double2 rb = rowb[buf][lane];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (warp == kw && q == kq) continue;
          const double2 c = make_double2(__shfl_sync(0xffffffffu, v[q].x, k), __shfl_sync(0xffffffffu, v[q].y, k));
          const double2 o = lane == k ? make_double2(0.0, 0.0) : v[q];
          v[q] = make_double2(fma(-c.x, rb.x, fma(c.y, rb.y, o.x)), fma(-c.x, rb.y, fma(-c.y, rb.x, o.y)));
        }
      }
#pragma unroll
    for (int q = 0; q < 4; ++q) Pbuf[(size_t)b * kNB * kNB + (4 * warp + q) * kNB + lane] = v[q];
    return;
  }
  const int u = blockIdx.x - nb, b = u / mtiles, mt = u % mtiles;
  const int row = t >> 1, half = t & 1, i = mt * 128 + row;
  const double2* src = A + (size_t)b * np * np + (size_t)i * np + k0 + 16 * half;
  double2 z[16];
  if (i >= k0 && i < k0 + kNB) {
#pragma unroll
    for (int c = 0; c < 16; ++c) z[c] = make_double2(16 * half + c == i - k0 ? -1.0 : 0.0, 0.0);
  } else {
#pragma unroll
    for (int c = 0; c < 16; ++c) z[c] = src[c];
  }
  unsigned m = 0;
#pragma unroll
  for (int c = 0; c < 16; ++c) m = max(m, max(mag_hi(z[c].x), mag_hi(z[c].y)));
  m = max(m, __shfl_xor_sync(0xffffffffu, m, 1));
  if (m >= 0x7ff00000u && status) atomicCAS(status, 0, DS_SINGULAR);  // not finite
  const int be = row_biased(m);
  if (half == 0) cexp[(size_t)b * np + i] = be - 1022;
  __nv_bfloat16* img = cimg + (size_t)u * kATile;
#pragma unroll
  for (int part = 0; part < 2; ++part)
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      long long y[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) y[c] = digit_word(part ? z[8 * g + c].y : z[8 * g + c].x, be);
      const int off = core_off(row, 32 * part + 16 * half + 8 * g);
      put_digits(y, [&](int s, uint4 v) { *reinterpret_cast<uint4*>(img + s * kARow + off) = v; });
    }
}

// ------------------------------------------------------------------ R panel

struct RSmem {
  static constexpr int kA = kATile * 2;          // digits of 128 columns of A_K
  static constexpr int kB = kS * 64 * kK * 2;    // digits of the 64 real rows of P
  static constexpr int kBytes = kA + kB + 1024;
};

// Digits of R = P A_{K,:} for 128 columns j of one matrix: thread (j = t & 127,
// h = t >> 7) cuts half of column j of A_K into digits (the MMA's A operand:
// rows j, k = [re | im]), all threads the rows of P (the B operand: row 2r =
// [Re P_r | -Im P_r], row 2r + 1 = [Im P_r | Re P_r]); 28 digit products give
// Re, Im of R[r][j] at lane j, columns 2r, 2r + 1 of seven orders; each thread
// turns 32 of its column's 64 sums into FP64 and those into the digits of the
// update's B operand: row 2j = [Re R_j | -Im R_j], row 2j + 1 = [Im R_j | Re R_j],
// one exponent per column.  A column costs the same whatever np is; at one CTA
// per SM the phases follow one another (latency bound), 4 % of the update's work.
__global__ void __launch_bounds__(256, 1)
    gj64_rpanel_kernel(const double2* __restrict__ A, int np, int k0, const double2* __restrict__ Pbuf,
                       __nv_bfloat16* __restrict__ rimg, int* __restrict__ rexp, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __nv_bfloat16* sa = reinterpret_cast<__nv_bfloat16*>(smem);
  __nv_bfloat16* sp = reinterpret_cast<__nv_bfloat16*>(smem + RSmem::kA);
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  __shared__ unsigned colmax[2][128];
  __shared__ int pexp[kNB];
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int b = blockIdx.y, j0 = blockIdx.x * 128, jl = t & 127, h = t >> 7, j = j0 + jl;
  constexpr uint32_t kCols = 512;  // 7 x 64
  if (t == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_barrier_init();
  }
  if (t < 128) colmax[0][t] = colmax[1][t] = 0;
  if (warp == 0) tmem_alloc(&tmem_slot, kCols);
  const double2* P = Pbuf + (size_t)b * kNB * kNB;
  double2 z[16];
  const double2* src = A + (size_t)b * np * np + (size_t)(k0 + 16 * h) * np + j;
#pragma unroll
  for (int c = 0; c < 16; ++c) z[c] = src[(size_t)c * np];
  {  // rows of P: eight threads per row, four entries each
    const int r = t >> 3, c4 = 4 * (t & 7);
    double2 p[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) p[c] = P[r * kNB + c4 + c];
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) m = max(m, max(mag_hi(p[c].x), mag_hi(p[c].y)));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int be = row_biased(m);
    if ((t & 7) == 0) pexp[r] = be - 1022;
    if (m >= 0x7ff00000u && status) atomicCAS(status, 0, DS_SINGULAR);
    long long y[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      y[c] = digit_word(p[c].x, be);
      y[4 + c] = digit_word(p[c].y, be);
    }
    const int o_re = core_off(2 * r, c4), o_im = core_off(2 * r, 32 + c4);  // row 2r + 1: 8 elements on
    put_digits(y, [&](int s, uint4 v) {
      __nv_bfloat16* d = sp + s * 64 * kK;
      const uint4 w = neg_bf16(v);
      *reinterpret_cast<uint2*>(d + o_re) = make_uint2(v.x, v.y);
      *reinterpret_cast<uint2*>(d + o_im) = make_uint2(w.z, w.w);
      *reinterpret_cast<uint2*>(d + o_re + 8) = make_uint2(v.z, v.w);
      *reinterpret_cast<uint2*>(d + o_im + 8) = make_uint2(v.x, v.y);
    });
  }
  tc_fence_before();
  __syncthreads();  // colmax cleared, TMEM allocated
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  {
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 16; ++c) m = max(m, max(mag_hi(z[c].x), mag_hi(z[c].y)));
    atomicMax(&colmax[0][jl], m);
  }
  __syncthreads();
  const unsigned cm = colmax[0][jl];
  if (cm >= 0x7ff00000u && h == 0 && status) atomicCAS(status, 0, DS_SINGULAR);
  const int be_a = row_biased(cm);
#pragma unroll
  for (int part = 0; part < 2; ++part)
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      long long y[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) y[c] = digit_word(part ? z[8 * g + c].y : z[8 * g + c].x, be_a);
      const int off = core_off(jl, 32 * part + 16 * h + 8 * g);
      put_digits(y, [&](int s, uint4 v) { *reinterpret_cast<uint4*>(sa + s * kARow + off) = v; });
    }
  fence_proxy_async();
  __syncthreads();
  if (t == 0) {
    for (int a = 0; a < kS; ++a)
      for (int n0 = 0; n0 < (kS - a) * 64; n0 += 256) {  // an MMA's N is at most 256
        const int n = (kS - a) * 64 - n0 < 256 ? (kS - a) * 64 - n0 : 256;
#pragma unroll
        for (int kk = 0; kk < kK / 16; ++kk)
          mma_bf16(tmem + (uint32_t)(a * 64 + n0), smem_desc(smem_u32(sa + a * kARow) + kk * 256, 128, 1024),
                   smem_desc(smem_u32(sp + n0 * kK) + kk * 256, 128, 1024), idesc_bf16(128, n),
                   (a > 0 || kk > 0) ? 1u : 0u);
      }
    mma_commit(&bar);
  }
  // the products read this CTA's shared memory: nobody leaves before they are done
  bool ok = mbar_wait(&bar, 0, &abort_flag);
  if (!ok) {
    const uint64_t t0 = global_ns();
    while (!mbar_test(&bar, 0) && global_ns() - t0 < kDrainNs) {
    }
  }
  ok = __syncthreads_and(ok);
  tc_fence_after();
  if (ok) {
    const int ebase = 1023 + (be_a - 1022) - 53;
    const bool in_k = j >= k0 && j < k0 + kNB;
    double2 rv[16];
#pragma unroll
    for (int g = 0; g < 4; ++g) {  // eight sums (four rows r) at a time
      float c[kS][8];
#pragma unroll
      for (int o = 0; o < kS; ++o)
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                     : "=f"(c[o][0]), "=f"(c[o][1]), "=f"(c[o][2]), "=f"(c[o][3]), "=f"(c[o][4]), "=f"(c[o][5]),
                       "=f"(c[o][6]), "=f"(c[o][7])
                     : "r"(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(o * 64 + 32 * h + 8 * g)));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int eb = ebase + pexp[16 * h + 4 * g + q];
        rv[4 * g + q].x = orders_to_double(c[0][2 * q], c[1][2 * q], c[2][2 * q], c[3][2 * q], c[4][2 * q],
                                           c[5][2 * q], c[6][2 * q], eb);
        rv[4 * g + q].y = orders_to_double(c[0][2 * q + 1], c[1][2 * q + 1], c[2][2 * q + 1], c[3][2 * q + 1],
                                           c[4][2 * q + 1], c[5][2 * q + 1], c[6][2 * q + 1], eb);
      }
    }
    if (in_k) {
#pragma unroll
      for (int r = 0; r < 16; ++r) rv[r] = P[(16 * h + r) * kNB + j - k0];
    }
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < 16; ++r) m = max(m, max(mag_hi(rv[r].x), mag_hi(rv[r].y)));
    atomicMax(&colmax[1][jl], m);
    __syncthreads();
    m = colmax[1][jl];
    if (m >= 0x7ff00000u && h == 0 && status) atomicCAS(status, 0, DS_SINGULAR);
    const int be = row_biased(m);
    if (h == 0) rexp[(size_t)b * np + j] = be - 1022;
    __nv_bfloat16* img = rimg + ((size_t)b * (np / kTn) + (j / kTn)) * kBTile;
    const int row = 2 * (j % kTn);
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      long long y[8];
      const int o_re = core_off(row, 16 * h + 8 * g), o_im = core_off(row, 32 + 16 * h + 8 * g);
#pragma unroll
      for (int c = 0; c < 8; ++c) y[c] = digit_word(rv[8 * g + c].x, be);
      put_digits(y, [&](int s, uint4 v) {
        *reinterpret_cast<uint4*>(img + s * kBDig + o_re) = v;
        *reinterpret_cast<uint4*>(img + s * kBDig + o_im + 8) = v;  // row 2j + 1
      });
#pragma unroll
      for (int c = 0; c < 8; ++c) y[c] = digit_word(rv[8 * g + c].y, be);
      put_digits(y, [&](int s, uint4 v) {
        *reinterpret_cast<uint4*>(img + s * kBDig + o_im) = neg_bf16(v);
        *reinterpret_cast<uint4*>(img + s * kBDig + o_re + 8) = v;
      });
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
  if (t == 0 && !ok && status) atomicCAS(status, 0, DS_TIMEOUT);
}

// ------------------------------------------------------------------ update

constexpr int kEpiW = 8;     // epilogue warps, two per TMEM lane quarter
constexpr int kBoxCols = 4;  // complex columns of a box (64 bytes per row), 32 rows
constexpr int kBoxBytes = 32 * kBoxCols * 16;
constexpr int kRing = 3;     // boxes of a warp: one worked on, two coming in or going out
struct USmem {
  static constexpr int kA = kATile * 2;
  static constexpr int kB = kBTile * 2;
  static constexpr int kBoxes = kEpiW * kRing * kBoxBytes;
  static constexpr int kBars = 512;
  static constexpr int kBytes = kA + 2 * kB + kBoxes + kBars + 1024;
};
struct UBars {
  uint64_t a_full, a_empty, b_full[2], b_empty[2], d_full[2], d_empty[2], drain;
  uint64_t box[kEpiW * kRing];
  uint32_t tmem_slot;
  int abort;
};
static_assert(sizeof(UBars) <= USmem::kBars, "barrier block");

__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  while (!mbar_test(bar, parity) && global_ns() - t0 < kDrainNs) {
  }
}

// Persistent over tiles of 128 rows x 16 complex columns, column tiles fastest,
// a contiguous run per CTA: the 112 KB of C digits stay in shared memory for a
// whole row tile, the 28 KB of R digits of the next tile come in behind the
// products (two buffers), two accumulator sets of 7 x 32 TMEM columns let the
// products of one tile run beside the epilogue of the other.  Warp 0 loads,
// warp 1 issues 28 MMAs per tile (7 digits x 4 k steps, N = 224 .. 32), warps
// 2-9 drain: a thread has one row and 8 complex columns, in two boxes of four.
// The old values come in by TMA two boxes ahead (64-byte swizzle: conflict-free
// 16-byte accesses with one row per lane), the result leaves by TMA from the
// same box.  Column tiles at or past `jskip` move up by `nskip` (a window that
// another kernel updates).
// What bounds it: the FP64 matrix is read and written once per 32 columns, 64 KB
// per tile, 3050 cycles at 6.5 TB/s over 152 SMs; the products take 1792, the
// epilogue about 1800 issue cycles, its FP64 subtraction 2048.
// With TMA FP64 reductions at L2 in place of load and subtract the payload rate
// measured 2.6 TB/s against 3.3 TB/s for read-modify-write: not used.
__global__ void __launch_bounds__(64 + 32 * kEpiW, 1)
    gj64_update_kernel(const __grid_constant__ CUtensorMap amap, int np, int mtiles, int ntn, int total, int k0,
                       int jskip, int nskip, const __nv_bfloat16* __restrict__ cimg, const int* __restrict__ cexp,
                       const __nv_bfloat16* __restrict__ rimg, const int* __restrict__ rexp, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  unsigned char* sa = smem;
  unsigned char* sb = smem + USmem::kA;
  unsigned char* sbox = sb + 2 * USmem::kB;
  UBars& bars = *reinterpret_cast<UBars*>(sbox + USmem::kBoxes);
  volatile int* abort_flag = &bars.abort;
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int lo = (int)((long long)blockIdx.x * total / gridDim.x);
  const int hi = (int)((long long)(blockIdx.x + 1) * total / gridDim.x);
  constexpr uint32_t kDCols = kS * 2 * kTn;  // 224
  constexpr uint32_t kCols = 512;
  if (t == 0) {
    mbar_init(&bars.a_full, 1);
    mbar_init(&bars.a_empty, 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(&bars.b_full[s], 1);
      mbar_init(&bars.b_empty[s], 1);
      mbar_init(&bars.d_full[s], 1);
      mbar_init(&bars.d_empty[s], kEpiW);
    }
    mbar_init(&bars.drain, 1);
    for (int k = 0; k < kEpiW * kRing; ++k) mbar_init(&bars.box[k], 1);
    bars.abort = 0;
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(&bars.tmem_slot, kCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars.tmem_slot;
  auto col_tile = [&](int jt) { return jt >= jskip ? jt + nskip : jt; };

  if (warp == 0) {
    if (lane == 0) {
      int na = 0, it = 0, cur = -1;
      for (int tile = lo; tile < hi; ++tile, ++it) {
        const int u = tile / ntn, jt = col_tile(tile % ntn);
        if (u != cur) {
          if (na > 0 && !mbar_wait(&bars.a_empty, (na - 1) & 1, abort_flag)) break;
          cur = u;
          ++na;
          mbar_arrive_expect_tx(&bars.a_full, USmem::kA);
          for (int s = 0; s < kS; ++s)
            bulk_g2s(sa + s * kTileBytes, cimg + (size_t)u * kATile + s * kARow, kTileBytes, &bars.a_full);
        }
        const int s = it & 1;
        if (it >= 2 && !mbar_wait(&bars.b_empty[s], ((it >> 1) - 1) & 1, abort_flag)) break;
        mbar_arrive_expect_tx(&bars.b_full[s], USmem::kB);
        bulk_g2s(sb + s * USmem::kB, rimg + ((size_t)(u / mtiles) * (np / kTn) + jt) * kBTile, USmem::kB,
                 &bars.b_full[s]);
      }
      // no copy may be in flight when the CTA leaves (after a failed wait)
      if (na > 0) drain_wait(&bars.a_full, (na - 1) & 1);
      const int n0 = (it + 1) / 2, n1 = it / 2;  // loads issued into buffers 0 and 1
      if (n0 > 0) drain_wait(&bars.b_full[0], (n0 - 1) & 1);
      if (n1 > 0) drain_wait(&bars.b_full[1], (n1 - 1) & 1);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      int na = 0, it = 0, cur = -1;
      for (int tile = lo; tile < hi; ++tile, ++it) {
        const int u = tile / ntn, s = it & 1;
        if (u != cur) {
          if (!mbar_wait(&bars.a_full, na & 1, abort_flag)) break;
          ++na;
          cur = u;
        }
        if (!mbar_wait(&bars.b_full[s], (it >> 1) & 1, abort_flag)) break;
        if (it >= 2 && !mbar_wait(&bars.d_empty[s], ((it >> 1) - 1) & 1, abort_flag)) break;
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)s * kDCols;
        const uint32_t ba = smem_u32(sb + s * USmem::kB);
#pragma unroll
        for (int a = 0; a < kS; ++a)
#pragma unroll
          for (int kk = 0; kk < kK / 16; ++kk)
            mma_bf16(d + (uint32_t)(a * 2 * kTn), smem_desc(smem_u32(sa + a * kTileBytes) + kk * 256, 128, 1024),
                     smem_desc(ba + kk * 256, 128, 1024), idesc_bf16(128, (kS - a) * 2 * kTn),
                     (a > 0 || kk > 0) ? 1u : 0u);
        mma_commit(&bars.b_empty[s]);
        mma_commit(&bars.d_full[s]);
        if (tile + 1 == hi || (tile + 1) / ntn != u) mma_commit(&bars.a_empty);
      }
      mma_commit(&bars.drain);
      drain_wait(&bars.drain, 0);
    }
  } else {
    const int w = warp - 2, quarter = warp & 3, c0 = 8 * (w >> 2);
    unsigned char* box0 = sbox + w * kRing * kBoxBytes;
    uint64_t* box_bar = bars.box + w * kRing;
    const int nbox = 2 * (hi - lo);
    // row and column of box k's corner in the batch's matrix of 2 np doubles per row
    auto corner = [&](int k, int& x, int& y) {
      const int tile = lo + (k >> 1), u = tile / ntn, jt = col_tile(tile % ntn);
      x = 2 * (jt * kTn + c0 + kBoxCols * (k & 1));
      y = (u / mtiles) * np + (u % mtiles) * 128 + quarter * 32;
    };
    auto fetch = [&](int k) {  // lane 0
      int x, y;
      corner(k, x, y);
      mbar_arrive_expect_tx(&box_bar[k % kRing], kBoxBytes);
      tma_load_2d(&amap, box0 + (k % kRing) * kBoxBytes, x, y, &box_bar[k % kRing]);
    };
    int issued = 0;
    if (lane == 0)
      for (; issued < 2 && issued < nbox; ++issued) fetch(issued);
    bool ok = true;
    for (int tile = lo, it = 0; tile < hi && ok; ++tile, ++it) {
      const int u = tile / ntn, jt = col_tile(tile % ntn), s = it & 1;
      const int b = u / mtiles, i = (u % mtiles) * 128 + quarter * 32 + lane;
      const bool ik = i >= k0 && i < k0 + kNB;  // the same for the whole warp
      const int ei = cexp[(size_t)b * np + i] + 1023 - 53;
      ok = __all_sync(0xffffffffu, mbar_wait(&bars.d_full[s], (it >> 1) & 1, abort_flag));
      if (!ok) break;
      tc_fence_after();
#pragma unroll 1
      for (int hb = 0; hb < 2 && ok; ++hb) {
        const int k = 2 * it + hb, slot = k % kRing, col = c0 + kBoxCols * hb, j = jt * kTn + col;
        const int4 ej = *reinterpret_cast<const int4*>(rexp + (size_t)b * np + j);
        float c[kS][8];
#pragma unroll
        for (int o = 0; o < kS; ++o)
          asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                       : "=f"(c[o][0]), "=f"(c[o][1]), "=f"(c[o][2]), "=f"(c[o][3]), "=f"(c[o][4]), "=f"(c[o][5]),
                         "=f"(c[o][6]), "=f"(c[o][7])
                       : "r"(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)s * kDCols +
                             (uint32_t)(o * 2 * kTn + 2 * col)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (hb == 1) {  // this warp is done with the accumulators
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bars.d_empty[s]);
        }
        ok = __all_sync(0xffffffffu, mbar_wait(&box_bar[slot], (k / kRing) & 1, abort_flag));
        if (!ok) break;
        const bool zero = ik || (j >= k0 && j < k0 + kNB);
        unsigned char* box = box0 + slot * kBoxBytes + lane * 64;
        const int sw = (lane >> 1) & 3;
        const int eq[4] = {ej.x, ej.y, ej.z, ej.w};
#pragma unroll
        for (int q = 0; q < kBoxCols; ++q) {
          double2* p = reinterpret_cast<double2*>(box + ((q ^ sw) << 4));
          const double2 old = zero ? make_double2(0.0, 0.0) : *p;
          const int eb = ei + eq[q];
          const double dx = orders_to_double(c[0][2 * q], c[1][2 * q], c[2][2 * q], c[3][2 * q], c[4][2 * q],
                                             c[5][2 * q], c[6][2 * q], eb);
          const double dy = orders_to_double(c[0][2 * q + 1], c[1][2 * q + 1], c[2][2 * q + 1], c[3][2 * q + 1],
                                             c[4][2 * q + 1], c[5][2 * q + 1], c[6][2 * q + 1], eb);
          *p = make_double2(old.x - dx, old.y - dy);
        }
        fence_proxy_async();
        __syncwarp();
        if (lane == 0) {
          int x, y;
          corner(k, x, y);
          tma_store_2d(&amap, box0 + slot * kBoxBytes, x, y);
          bulk_commit();
          if (issued < nbox) {
            bulk_wait_read_n<1>();  // the store from the slot that is filled next has read it
            fetch(issued++);
          }
        }
        __syncwarp();
      }
    }
    if (lane == 0) {
      // every box load issued has landed (on the normal path they all were waited for)
      for (int k = issued > kRing ? issued - kRing : 0; k < issued; ++k) drain_wait(&box_bar[k % kRing], (k / kRing) & 1);
      bulk_wait_all();
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kCols);
  }
  if (t == 0 && bars.abort && status) atomicCAS(status, 0, DS_TIMEOUT);
}

// The batch as one tensor of 2 np doubles per row, moved in boxes of four complex columns x 32 rows.
int encode_f64_boxes(CUtensorMap* map, double2* base, uint64_t np, uint64_t rows) {
  using Fn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                          const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                          CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
  static const Fn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<Fn>(f);
  }();
  if (!fn) return set_error(NEDMFT_ECUDA, "cuTensorMapEncodeTiled is not available from the CUDA driver");
  const cuuint64_t dims[2] = {2 * np, rows};
  const cuuint64_t strides[1] = {2 * np * sizeof(double)};
  const cuuint32_t box[2] = {2 * kBoxCols, 32};
  const cuuint32_t elem_strides[2] = {1, 1};
  const CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 2, base, dims, strides, box, elem_strides,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(NEDMFT_ECUDA, "cuTensorMapEncodeTiled (FP64) failed (CUresult %d)", (int)r);
  return NEDMFT_OK;
}

struct Gj64Layout {
  size_t p, c, r, ce, re, total;
};
Gj64Layout gj64_layout(int np, int nb) {
  Gj64Layout L;
  const size_t n = np, b = nb;
  L.p = align256(sizeof(double2) * kNB * kNB * b);
  L.c = align256(2 * (size_t)kATile * (n / 128) * b);
  L.r = align256(2 * (size_t)kBTile * (n / kTn) * b);
  L.ce = align256(sizeof(int) * n * b);
  L.re = align256(sizeof(int) * n * b);
  L.total = L.p + L.c + L.r + L.ce + L.re;
  return L;
}

}  // namespace

size_t gj64_scratch_bytes(int np, int nb) { return gj64_layout(np, nb).total; }

int gj64_set_wait_ns(uint64_t ns, cudaStream_t st) {
  NED_CUDA(cudaMemcpyToSymbolAsync(umma::g_wait_ns, &ns, sizeof(ns), 0, cudaMemcpyHostToDevice, st));
  NED_CUDA(cudaStreamSynchronize(st));
  return NEDMFT_OK;
}

// In-place inverses of nb matrices (np x np, np a multiple of 128, identity
// outside n x n) with `scratch` of gj64_scratch_bytes(np, nb).  Blocks of 32
// columns past n are the identity's: their steps, and the column tiles past n,
// change nothing and are left out.
int gj64_invert(double2* A, int n, int np, int nb, void* scratch, int* status, cudaStream_t st) {
  if (np % 128) return set_error(NEDMFT_EINVAL, "gj64_invert: np = %d not a multiple of 128", np);
  const Gj64Layout L = gj64_layout(np, nb);
  char* p = static_cast<char*>(scratch);
  double2* pbuf = reinterpret_cast<double2*>(p); p += L.p;
  __nv_bfloat16* cimg = reinterpret_cast<__nv_bfloat16*>(p); p += L.c;
  __nv_bfloat16* rimg = reinterpret_cast<__nv_bfloat16*>(p); p += L.r;
  int* cexp = reinterpret_cast<int*>(p); p += L.ce;
  int* rexp = reinterpret_cast<int*>(p);
  CUtensorMap map;
  int rc = encode_f64_boxes(&map, A, np, (uint64_t)np * nb);
  int sms = 0;
  if (!rc) rc = device_sm_count(&sms);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_rpanel_kernel), RSmem::kBytes);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_update_kernel), USmem::kBytes);
  if (rc) return rc;
  const int mtiles = np / 128, ntn = ceil_div(n, kTn), total = nb * mtiles * ntn;
  for (int k0 = 0; k0 < n; k0 += kNB) {
    gj64_pivot_kernel<<<nb + nb * mtiles, 256, 0, st>>>(A, np, mtiles, k0, nb, pbuf, cimg, cexp, status);
    NED_LAUNCH_CHECK("gj64_pivot_kernel");
    gj64_rpanel_kernel<<<dim3(mtiles, nb), 256, RSmem::kBytes, st>>>(A, np, k0, pbuf, rimg, rexp, status);
    NED_LAUNCH_CHECK("gj64_rpanel_kernel");
    const int slot = instr_begin(st);
    gj64_update_kernel<<<total < sms ? total : sms, 64 + 32 * kEpiW, USmem::kBytes, st>>>(
        map, np, mtiles, ntn, total, k0, ntn, 0, cimg, cexp, rimg, rexp, status);
    NED_LAUNCH_CHECK("gj64_update_kernel");
    const int live = n - k0 < kNB ? n - k0 : kNB;
    instr_end(slot, st, 8.0 * (double)n * n * live * nb, 2.0 * sizeof(double2) * (double)n * n * nb);
  }
  return NEDMFT_OK;
}

}  // namespace nedmft
