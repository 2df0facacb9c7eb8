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
constexpr int kPTile = kS * 64 * kK;         // ... of the 64 real rows of P

__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  while (!mbar_test(bar, parity) && global_ns() - t0 < kDrainNs) {
  }
}
// eight TMEM columns of this warp's 32 lanes (wait with tmem_wait_ld)
__device__ __forceinline__ void tmem_ld8(uint32_t addr, float (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "r"(addr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

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
template <int S = 0, class Put>
__device__ __forceinline__ void put_digits2(const long long (&y)[16], Put&& put) {
  put(S, make_uint4(digit_pair<S>(y[0], y[1]), digit_pair<S>(y[2], y[3]), digit_pair<S>(y[4], y[5]),
                    digit_pair<S>(y[6], y[7])),
      make_uint4(digit_pair<S>(y[8], y[9]), digit_pair<S>(y[10], y[11]), digit_pair<S>(y[12], y[13]),
                 digit_pair<S>(y[14], y[15])));
  if constexpr (S + 1 < kS) put_digits2<S + 1>(y, put);
}
// 32 bytes (one sector) in one store; p 32-byte aligned
__device__ __forceinline__ void st32(void* p, uint4 a, uint4 b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
               "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}
__device__ __forceinline__ uint4 neg_bf16(uint4 v) {
  return make_uint4(v.x ^ 0x80008000u, v.y ^ 0x80008000u, v.z ^ 0x80008000u, v.w ^ 0x80008000u);
}
// element offset of (row, k) in a canonical K-major tile of 64 k
__device__ __forceinline__ int core_off(int row, int k) { return ((row >> 3) * 8 + (k >> 3)) * 64 + (row & 7) * 8 + (k & 7); }

// ------------------------------------------------------------------ order sums to FP64

// 2^(e-53) sum_o c_o 2^(8(5-o)) / 2 as a double, rounded once; c_o, o = 0 .. 6,
// are integers with |c_o| <= (o + 1) 2^20.  ebase = 1023 + e - 53.
// Float to int by adding 1.5 2^23 (below 2^22; conversion instructions run at
// an eighth of the rate), orders 4 .. 6 with the half of order 4 split off
// first.  Pairs of orders share a word, offset so that it stays positive, and
// three wide multiply-adds make the sum T, 64 bits, in units of 2.  Its leading
// bit comes from a float rounded towards zero; then it is shifted, rounded and
// assembled on the integer units: about 40 instructions, none in FP64.  Written
// as single instructions, without a branch: the same in C++ with 64-bit shifts
// and conditionals took twice as many.
__device__ __forceinline__ double orders_to_double(float c0, float c1, float c2, float c3, float c4, float c5,
                                                   float c6, int ebase) {
  constexpr float kM = 12582912.f;
  constexpr unsigned long long kOff = 0x8B400000ull;  // 0x4B400000 * 257 mod 2^32: the offset of a pair's word
  constexpr unsigned long long kLess = 0ull - kOff * ((1ull << 31) + (1ull << 15) + 1ull);
  const uint32_t b0 = __float_as_uint(c0 + kM), b1 = __float_as_uint(c1 + kM);
  const uint32_t b2 = __float_as_uint(c2 + kM), b3 = __float_as_uint(c3 + kM);
  const float t4 = fmaf(c4, 0.5f, kM);
  const float rem = fmaf(c4, 0.5f, kM - t4);
  const float g = fmaf(rem, 512.f, fmaf(c6, 0.00390625f, c5));
  const uint32_t b4 = __float_as_uint(t4), b5 = __float_as_uint(fmaf(g, 0.5f, kM));
  const uint32_t u0 = b0 * 256u + b1, u1 = b2 * 256u + b3, u2 = b4 * 256u + b5;  // the pairs + kOff
  uint32_t rh, ql;
  asm("{\n\t"
      ".reg .u64 t;\n\t.reg .u32 lo, hi, s, n, ld, e, qh;\n\t.reg .f32 fh, fl;\n\t.reg .pred z;\n\t"
      "mad.wide.u32 t, %4, 1, %5;\n\t"
      "mad.wide.u32 t, %3, 32768, t;\n\t"
      "mad.wide.u32 t, %2, 0x80000000, t;\n\t"
      "mov.b64 {lo, hi}, t;\n\t"
      "shr.s32 s, hi, 31;\n\t"  // |T|
      "xor.b32 lo, lo, s;\n\txor.b32 hi, hi, s;\n\t"
      "sub.cc.u32 lo, lo, s;\n\tsubc.u32 hi, hi, s;\n\t"
      "cvt.rz.f32.u32 fh, hi;\n\tcvt.rz.f32.u32 fl, lo;\n\t"
      "fma.rz.f32 fh, fh, 0f4F800000, fl;\n\t"
      "mov.b32 ld, fh;\n\tshr.u32 ld, ld, 23;\n\t"  // 127 + index of the leading bit, 0 for T = 0
      "sub.u32 n, 189, ld;\n\t"
      "mov.b64 t, {lo, hi};\n\tshl.b64 t, t, n;\n\tmov.b64 {lo, hi}, t;\n\t"  // leading bit to bit 62
      "add.cc.u32 lo, lo, 0x200;\n\taddc.u32 hi, hi, 0;\n\t"                    // 53 bits, rounded to nearest
      "shf.r.wrap.b32 %1, lo, hi, 10;\n\tshr.u32 qh, hi, 10;\n\t"
      "add.s32 e, ld, %6;\n\tmin.s32 e, e, 2046;\n\t"  // beyond FP64: infinite or NaN, caught at the next digit cut
      "mad.lo.u32 qh, e, 0x100000, qh;\n\t"
      "and.b32 s, s, 0x80000000;\n\tor.b32 qh, qh, s;\n\t"
      "setp.eq.u32 z, ld, 0;\n\tselp.u32 %0, 0, qh, z;\n\t"
      "}"
      : "=&r"(rh), "=&r"(ql)
      : "r"(u0), "r"(u1), "r"(u2), "l"(kLess), "r"(ebase - 128));
  return __hiloint2double((int)rh, (int)ql);
}

// ------------------------------------------------------------------ pivot block and C digits

// 1 / z as cinv_guard, the real reciprocal by two Newton steps on the
// hardware's approximation (20 bits, then 40, then all): a third of the FP64
// instructions of a division on the pivot row's serial path.
__device__ __forceinline__ bool recip(double2 z, double2& out) {
  const double m = z.x * z.x + z.y * z.y;
  if (!(m > 1e-24)) {  // |z| <= 1e-12 or NaN
    out = make_double2(1e12, 0.0);
    return false;
  }
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(m));
  r = fma(r, fma(-m, r, 1.0), r);
  r = fma(r, fma(-m, r, 1.0), r);
  out = make_double2(z.x * r, -z.y * r);
  return true;
}

// CTAs 0 .. nb-1: P = inv(A_KK) of matrix b, 32 x 32 FP64, a warp per four
// rows, lane = column.  Step k: the pivot row, divided by its pivot (its own
// entry replaced by the pivot's inverse), is in shared memory (two buffers, one
// barrier per step); every other row subtracts its entry of column k times it,
// that entry counted as zero before.  The warp of the next pivot row takes that
// row first and publishes it, so the reciprocal is off the other warps' path.
// FP64 bound: 32 rows x 4 FMAs x 16 cycles per step, 33 us.
// CTAs nb ..: digits of 128 rows of C, two threads per row; this work hides
// behind the pivot blocks' latency.
__global__ void __launch_bounds__(256) gj64_pivot_kernel(const double2* __restrict__ A, int np, int mtiles, int k0,
                                                         int nb, double2* __restrict__ Pbuf,
                                                         __nv_bfloat16* __restrict__ pimg, int* __restrict__ pexp,
                                                         __nv_bfloat16* __restrict__ cimg, int* __restrict__ cexp,
                                                         int* status) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  if ((int)blockIdx.x < nb) {
    __shared__ double2 rowb[2][32];
    __shared__ double2 prow[kNB][kNB + 1];
    const int b = blockIdx.x;
    const double2* a = A + (size_t)b * np * np + (size_t)k0 * np + k0;
    double2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = a[(size_t)(4 * warp + q) * np + lane];
    // row (warp, kq) as step k's pivot row: divided by its pivot and published
    auto publish = [&](double2& z, int k) {
      const double2 d = make_double2(__shfl_sync(0xffffffffu, z.x, k), __shfl_sync(0xffffffffu, z.y, k));
      double2 pinv;
      if (!recip(d, pinv) && lane == 0 && status) atomicCAS(status, 0, DS_SINGULAR);
      z = lane == k ? pinv : cmul(z, pinv);
      rowb[k & 1][lane] = z;
    };
    if (warp == 0) publish(v[0], 0);
    __syncthreads();
    for (int kw = 0; kw < 8; ++kw)
#pragma unroll
      for (int kq = 0; kq < 4; ++kq) {
        const int k = 4 * kw + kq;
        const double2 rb = rowb[k & 1][lane];
        auto eliminate = [&](double2& z) {
          const double2 c = make_double2(__shfl_sync(0xffffffffu, z.x, k), __shfl_sync(0xffffffffu, z.y, k));
          const double2 o = lane == k ? make_double2(0.0, 0.0) : z;
          z = make_double2(fma(-c.x, rb.x, fma(c.y, rb.y, o.x)), fma(-c.x, rb.y, fma(-c.y, rb.x, o.y)));
        };
        constexpr int kNext[4] = {1, 2, 3, 0};  // the next pivot row's place in its warp
        const int nq = kNext[kq];
        const bool mine = k + 1 < 32 && warp == (kq == 3 ? kw + 1 : kw);
        if (mine) {  // the next pivot row first: its reciprocal runs beside the other warps' rows
          eliminate(v[nq]);
          publish(v[nq], k + 1);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (!(warp == kw && q == kq) && !(mine && q == nq)) eliminate(v[q]);
        __syncthreads();
      }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = 4 * warp + q;
      Pbuf[(size_t)b * kNB * kNB + r * kNB + lane] = v[q];
      prow[r][lane] = v[q];
    }
    __syncthreads();
    // digits of the 64 real rows of P, eight threads per row r, four entries
    // each: row 2r = [Re P_r | -Im P_r], row 2r + 1 = [Im P_r | Re P_r]
    const int r = t >> 3, c4 = 4 * (t & 7);
    double2 p[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) p[c] = prow[r][c4 + c];
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) m = max(m, max(mag_hi(p[c].x), mag_hi(p[c].y)));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    const int be = row_biased(m);
    if ((t & 7) == 0) pexp[b * kNB + r] = be - 1022;
    if (m >= 0x7ff00000u && status) atomicCAS(status, 0, DS_SINGULAR);
    long long y[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      y[c] = digit_word(p[c].x, be);
      y[4 + c] = digit_word(p[c].y, be);
    }
    const int o_re = core_off(2 * r, c4), o_im = core_off(2 * r, 32 + c4);  // row 2r + 1: 8 elements on
    put_digits(y, [&](int s, uint4 w) {
      __nv_bfloat16* d = pimg + (size_t)b * kPTile + s * 64 * kK;
      const uint4 n = neg_bf16(w);
      *reinterpret_cast<uint2*>(d + o_re) = make_uint2(w.x, w.y);
      *reinterpret_cast<uint2*>(d + o_im) = make_uint2(n.z, n.w);
      *reinterpret_cast<uint2*>(d + o_re + 8) = make_uint2(w.z, w.w);
      *reinterpret_cast<uint2*>(d + o_im + 8) = make_uint2(w.x, w.y);
    });
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
  static constexpr int kA = kATile * 2;  // digits of 128 columns of A_K
  static constexpr int kB = kPTile * 2;  // digits of the 64 real rows of P
  static constexpr int kBytes = kA + kB + 1024;
};

// Digits of R = P A_{K,:} for 128 columns j of one matrix: thread (j = t & 127,
// h = t >> 7) cuts a quarter of column j of A_K into digits (the MMA's A
// operand: rows j, k = [re | im]) while the digits of P come in (the B
// operand); 28 digit products give Re, Im of R[r][j] at lane j, columns 2r,
// 2r + 1 of seven orders; each thread turns 16 of its column's 64 sums into
// FP64 and those into the digits of the update's B operand: row 2j =
// [Re R_j | -Im R_j], row 2j + 1 = [Im R_j | Re R_j], one exponent per column.
// One CTA per SM, its phases one after the other: latency bound, hence 16 warps.
__global__ void __launch_bounds__(512, 1)
    gj64_rpanel_kernel(const double2* __restrict__ A, int np, int k0, const double2* __restrict__ Pbuf,
                       const __nv_bfloat16* __restrict__ pimg, const int* __restrict__ pexp,
                       __nv_bfloat16* __restrict__ rimg, int* __restrict__ rexp, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  __nv_bfloat16* sa = reinterpret_cast<__nv_bfloat16*>(smem);
  __nv_bfloat16* sp = reinterpret_cast<__nv_bfloat16*>(smem + RSmem::kA);
  __shared__ __align__(8) uint64_t bars[2];  // the digits of P, the products
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int abort_flag;
  __shared__ unsigned colmax[2][128];
  const int t = threadIdx.x, warp = t >> 5;
  const int b = blockIdx.y, j0 = blockIdx.x * 128, jl = t & 127, h = t >> 7, j = j0 + jl;
  constexpr uint32_t kCols = 512;  // 7 x 64
  if (t == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&bars[1], 1);
    abort_flag = 0;
    fence_barrier_init();
    mbar_arrive_expect_tx(&bars[0], RSmem::kB);
    bulk_g2s(sp, pimg + (size_t)b * kPTile, RSmem::kB, &bars[0]);
  }
  if (t < 128) colmax[0][t] = colmax[1][t] = 0;
  if (warp == 0) tmem_alloc(&tmem_slot, kCols);
  double2 z[8];
  const double2* src = A + (size_t)b * np * np + (size_t)(k0 + 8 * h) * np + j;
#pragma unroll
  for (int c = 0; c < 8; ++c) z[c] = src[(size_t)c * np];
  tc_fence_before();
  __syncthreads();  // barriers, colmax, TMEM address
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  {
    unsigned m = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) m = max(m, max(mag_hi(z[c].x), mag_hi(z[c].y)));
    atomicMax(&colmax[0][jl], m);
  }
  __syncthreads();
  const unsigned cm = colmax[0][jl];
  if (cm >= 0x7ff00000u && h == 0 && status) atomicCAS(status, 0, DS_SINGULAR);
  const int be_a = row_biased(cm);
#pragma unroll
  for (int part = 0; part < 2; ++part) {
    long long y[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) y[c] = digit_word(part ? z[c].y : z[c].x, be_a);
    const int off = core_off(jl, 32 * part + 8 * h);
    put_digits(y, [&](int s, uint4 v) { *reinterpret_cast<uint4*>(sa + s * kARow + off) = v; });
  }
  fence_proxy_async();
  bool ok = mbar_wait(&bars[0], 0, &abort_flag);
  if (!ok) drain_wait(&bars[0], 0);
  ok = __syncthreads_and(ok);
  if (t == 0) {
    tc_fence_after();
    if (ok)
      for (int a = 0; a < kS; ++a)
        for (int n0 = 0; n0 < (kS - a) * 64; n0 += 256) {  // an MMA's N is at most 256
          const int n = (kS - a) * 64 - n0 < 256 ? (kS - a) * 64 - n0 : 256;
#pragma unroll
          for (int kk = 0; kk < kK / 16; ++kk)
            mma_bf16(tmem + (uint32_t)(a * 64 + n0), smem_desc(smem_u32(sa + a * kARow) + kk * 256, 128, 1024),
                     smem_desc(smem_u32(sp + n0 * kK) + kk * 256, 128, 1024), idesc_bf16(128, n),
                     (a > 0 || kk > 0) ? 1u : 0u);
        }
    mma_commit(&bars[1]);
  }
  // the products read this CTA's shared memory: nobody leaves before they are done
  if (ok) ok = mbar_wait(&bars[1], 0, &abort_flag);
  if (!ok) drain_wait(&bars[1], 0);
  ok = __syncthreads_and(ok);
  tc_fence_after();
  if (ok) {
    const int ebase = 1023 + (be_a - 1022) - 53;
    const double2* P = Pbuf + (size_t)b * kNB * kNB;
    double2 rv[8];
#pragma unroll 1
    for (int g = 0; g < 2; ++g) {  // eight sums (four rows r) at a time
      float c[kS][8];
#pragma unroll
      for (int o = 0; o < kS; ++o)
        tmem_ld8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(o * 64 + 16 * h + 8 * g), c[o]);
      tmem_wait_ld();
      double2 x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int eb = ebase + pexp[b * kNB + 8 * h + 4 * g + q];
        x[q].x = orders_to_double(c[0][2 * q], c[1][2 * q], c[2][2 * q], c[3][2 * q], c[4][2 * q], c[5][2 * q],
                                  c[6][2 * q], eb);
        x[q].y = orders_to_double(c[0][2 * q + 1], c[1][2 * q + 1], c[2][2 * q + 1], c[3][2 * q + 1],
                                  c[4][2 * q + 1], c[5][2 * q + 1], c[6][2 * q + 1], eb);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) (g ? rv[4 + q] : rv[q]) = x[q];
    }
    if (j >= k0 && j < k0 + kNB) {
#pragma unroll
      for (int r = 0; r < 8; ++r) rv[r] = P[(8 * h + r) * kNB + j - k0];
    }
    unsigned m = 0;
#pragma unroll
    for (int r = 0; r < 8; ++r) m = max(m, max(mag_hi(rv[r].x), mag_hi(rv[r].y)));
    atomicMax(&colmax[1][jl], m);
    __syncthreads();
    m = colmax[1][jl];
    if (m >= 0x7ff00000u && h == 0 && status) atomicCAS(status, 0, DS_SINGULAR);
    const int be = row_biased(m);
    if (h == 0) rexp[(size_t)b * np + j] = be - 1022;
    __nv_bfloat16* img = rimg + ((size_t)b * (np / kTn) + (j / kTn)) * kBTile;
    const int row = 2 * (j % kTn);
    const int o_re = core_off(row, 8 * h), o_im = core_off(row, 32 + 8 * h);  // row 2j + 1: 8 elements on
    long long y[16];  // Re and Im: rows 2j and 2j + 1 lie side by side, 32 bytes to a store
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      y[c] = digit_word(rv[c].x, be);
      y[8 + c] = digit_word(rv[c].y, be);
    }
    put_digits2(y, [&](int s, uint4 re, uint4 im) {
      st32(img + s * kBDig + o_re, re, im);
      st32(img + s * kBDig + o_im, neg_bf16(im), re);
    });
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
constexpr int kBoxCols = 8;  // complex columns of a box (128 bytes per row), 32 rows
constexpr int kBoxBytes = 32 * kBoxCols * 16;
struct USmem {
  static constexpr int kA = kATile * 2;
  static constexpr int kB = kBTile * 2;
  static constexpr int kBoxes = kEpiW * kBoxBytes;
  static constexpr int kBars = 512;
  static constexpr int kBytes = kA + 2 * kB + kBoxes + kBars + 1024;
};
struct UBars {
  uint64_t a_full, a_empty, b_full[2], b_empty[2], d_full[2], d_empty[2], drain;
  uint32_t tmem_slot;
  int abort;
};
static_assert(sizeof(UBars) <= USmem::kBars, "barrier block");

// Persistent over tiles of 128 rows x 16 complex columns, column tiles fastest,
// a contiguous run per CTA: the 112 KB of C digits stay in shared memory for a
// whole row tile, the 28 KB of R digits of the next tile come in behind the
// products (two buffers), two accumulator sets of 7 x 32 TMEM columns let the
// products of one tile run beside the epilogue of the other.  Warp 0 loads,
// warp 1 issues 28 MMAs per tile (7 digits x 4 k steps, N = 224 .. 32), warps
// 2-9 drain: a thread has one row and 8 complex columns, a warp one box of 32
// rows x 128 bytes, which is added to A at L2 by a TMA FP64 reduction (rows and
// columns of block K: stored).  Column tiles at or past `jskip` move up by
// `nskip` (a window that another kernel updates).
// What bounds it: the L2's FP64 reductions, 2.6 TB/s of payload measured alone;
// here 604 MB (64 matrices of 768 x 768) in 243 us, 2.5 TB/s.  Products 1792
// cycles per tile of 4400, epilogue about 1700 issue cycles.  Measured before
// it: old values loaded by TMA in 64-byte rows two boxes ahead, subtracted and
// stored, 292 us (the shared memory left for boxes does not cover the latency);
// half of the boxes each way, 274 us.
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
    unsigned char* box = sbox + w * kBoxBytes;
    // tile coordinates: column tile, matrix, row tile; stepped, not divided
    struct Pos {
      int jn, b, mt;
    };
    auto step = [&](Pos& p) {
      if (++p.jn == ntn) {
        p.jn = 0;
        if (++p.mt == mtiles) {
          p.mt = 0;
          ++p.b;
        }
      }
    };
    Pos cur{lo % ntn, lo / ntn / mtiles, lo / ntn % mtiles};
    bool ok = true;
    for (int tile = lo, it = 0; tile < hi && ok; ++tile, ++it) {
      const int jt = col_tile(cur.jn), s = it & 1;
      const int b = cur.b, i = cur.mt * 128 + quarter * 32 + lane;
      const bool ik = i >= k0 && i < k0 + kNB;  // the same for the whole warp
      const int ei = cexp[(size_t)b * np + i] + 1023 - 53;
      ok = __all_sync(0xffffffffu, mbar_wait(&bars.d_full[s], (it >> 1) & 1, abort_flag));
      if (!ok) break;
      tc_fence_after();
      // the warp's sums at once: the accumulators are free for the next tile's products before the arithmetic
      float acc[2][kS][8];
#pragma unroll
      for (int hb = 0; hb < 2; ++hb)
#pragma unroll
        for (int o = 0; o < kS; ++o)
          tmem_ld8(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)s * kDCols +
                       (uint32_t)(o * 2 * kTn + 2 * c0 + 8 * hb),
                   acc[hb][o]);
      tmem_wait_ld();
      tc_fence_before();
      if (lane == 0) bulk_wait_read_n<0>();  // the last tile's box has been read
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars.d_empty[s]);
      const int j = jt * kTn + c0;
#pragma unroll
      for (int hb = 0; hb < 2; ++hb) {
        const int4 ej = *reinterpret_cast<const int4*>(rexp + (size_t)b * np + j + 4 * hb);
        const int eq[4] = {ej.x, ej.y, ej.z, ej.w};
        const float(&c)[kS][8] = acc[hb];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int eb = ei + eq[q];
          const double dx = orders_to_double(c[0][2 * q], c[1][2 * q], c[2][2 * q], c[3][2 * q], c[4][2 * q],
                                             c[5][2 * q], c[6][2 * q], eb);
          const double dy = orders_to_double(c[0][2 * q + 1], c[1][2 * q + 1], c[2][2 * q + 1], c[3][2 * q + 1],
                                             c[4][2 * q + 1], c[5][2 * q + 1], c[6][2 * q + 1], eb);
          *reinterpret_cast<double2*>(box + lane * 128 + (((4 * hb + q) ^ (lane & 7)) << 4)) = make_double2(-dx, -dy);
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0) {
        const int x = 2 * j, y = b * np + cur.mt * 128 + quarter * 32;
        if (ik || (j >= k0 && j < k0 + kNB)) tma_store_2d(&amap, box, x, y);  // block K: nothing to add to
        else tma_reduce_add_2d(&amap, box, x, y);
        bulk_commit();
      }
      __syncwarp();
      step(cur);
    }
    if (lane == 0) bulk_wait_all();
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
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return set_error(NEDMFT_ECUDA, "cuTensorMapEncodeTiled (FP64) failed (CUresult %d)", (int)r);
  return NEDMFT_OK;
}

struct Gj64Layout {
  size_t p, pi, pe, c, r, ce, re, total;
};
Gj64Layout gj64_layout(int np, int nb) {
  Gj64Layout L;
  const size_t n = np, b = nb;
  L.p = align256(sizeof(double2) * kNB * kNB * b);
  L.pi = align256(2 * (size_t)kPTile * b);
  L.pe = align256(sizeof(int) * kNB * b);
  L.c = align256(2 * (size_t)kATile * (n / 128) * b);
  L.r = align256(2 * (size_t)kBTile * (n / kTn) * b);
  L.ce = align256(sizeof(int) * n * b);
  L.re = align256(sizeof(int) * n * b);
  L.total = L.p + L.pi + L.pe + L.c + L.r + L.ce + L.re;
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
  __nv_bfloat16* pimg = reinterpret_cast<__nv_bfloat16*>(p); p += L.pi;
  int* pexp = reinterpret_cast<int*>(p); p += L.pe;
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
    gj64_pivot_kernel<<<nb + nb * mtiles, 256, 0, st>>>(A, np, mtiles, k0, nb, pbuf, pimg, pexp, cimg,
                                                          cexp, status);
    NED_LAUNCH_CHECK("gj64_pivot_kernel");
    gj64_rpanel_kernel<<<dim3(mtiles, nb), 512, RSmem::kBytes, st>>>(A, np, k0, pbuf, pimg, pexp, rimg, rexp,
                                                                        status);
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
