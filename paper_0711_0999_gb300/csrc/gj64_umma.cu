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
// The 28 products of order <= 6 are kept (each left out is below 2^-56 of the row
// and column maxima, all of them together about 2^-53), their sums are put together
// in 64-bit integers and rounded once to FP64.  The whole inversion errs less than
// in FP64 FMAs (figures at refined_inverse).
//
// One MMA per digit a of the left operand takes all its partners b = 0 .. 6-a
// at once: the right operand's digits lie back to back in shared memory, and
// orders a .. 6 back to back in TMEM.
#include <stddef.h>

#include <type_traits>

#include "lattice.cuh"
#include "umma_core.cuh"

namespace nedmft {

using namespace umma;

namespace {

constexpr int kS = 7;    // digits of an operand, orders kept
constexpr int kO = 8;    // orders of the pivot blocks' residuals
constexpr int kNB = 32;  // complex columns per step
constexpr int kK = 64;   // reals per row of C and column of R: [re | im]
constexpr int kTn = 16;  // complex columns of an update tile
constexpr int kARow = kTileElems;            // bf16 elements of one digit of a 128-row tile
constexpr int kATile = kS * kTileElems;      // ... of all digits
constexpr int kBDig = 2 * kTn * kK;          // bf16 elements of one digit of a 16-column tile of R
constexpr int kBTile = kS * kBDig;
constexpr int kPTile = kS * 64 * kK;         // ... of the 64 real rows of P

// shared -> global bulk copy and FP64 reduction (add at L2), tracked by bulk groups
__device__ __forceinline__ void bulk_store(double2* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_add_f64(double2* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f64 [%0], [%1], %2;" ::"l"(dst),
               "r"(smem_u32(src)), "r"(bytes)
               : "memory");
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

constexpr unsigned long long kPairOff = 0x8B400000ull;  // 0x4B400000 * 257 mod 2^32: the offset of a pair's word
constexpr unsigned long long kLess = 0ull - kPairOff * ((1ull << 31) + (1ull << 15) + 1ull);
// the orders in pairs, each word kPairOff above its value: T = u0 2^31 + u1 2^15 + u2 + kLess
__device__ __forceinline__ void order_words(float c0, float c1, float c2, float c3, float c4, float c5, float c6,
                                            uint32_t& u0, uint32_t& u1, uint32_t& u2) {
  constexpr float kM = 12582912.f;
  const uint32_t b0 = __float_as_uint(c0 + kM), b1 = __float_as_uint(c1 + kM);
  const uint32_t b2 = __float_as_uint(c2 + kM), b3 = __float_as_uint(c3 + kM);
  const float t4 = fmaf(c4, 0.5f, kM);
  const float rem = fmaf(c4, 0.5f, kM - t4);
  const float g = fmaf(rem, 512.f, fmaf(c6, 0.00390625f, c5));
  const uint32_t b4 = __float_as_uint(t4), b5 = __float_as_uint(fmaf(g, 0.5f, kM));
  u0 = b0 * 256u + b1;
  u1 = b2 * 256u + b3;
  u2 = b4 * 256u + b5;
}

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
  uint32_t u0, u1, u2;
  order_words(c0, c1, c2, c3, c4, c5, c6, u0, u1, u2);
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

// The same sum plus `more` (in its units) and with order 7, as a float of about 24 bits, times
// `scale`.  Orders 6 and 7 and what a unit cannot hold are added to the sum of the others as
// a float: a sum that cancels down to a few units keeps ten more bits.
__device__ __forceinline__ float orders_to_float(float c0, float c1, float c2, float c3, float c4, float c5, float c6,
                                                 float c7, unsigned long long more, float scale) {
  constexpr float kM = 12582912.f;
  uint32_t u0, u1, u2;
  order_words(c0, c1, c2, c3, c4, c5, 0.f, u0, u1, u2);
  const float h4 = fmaf(c4, 0.5f, kM) - kM;
  const float g = fmaf(fmaf(c4, 0.5f, -h4), 512.f, c5);                        // as order_words has it
  const float frac = fmaf(g, 0.5f, -(fmaf(g, 0.5f, kM) - kM));                 // 0 or +-1/2
  const float low = frac + fmaf(c7, 7.62939453125e-6f, c6 * 0.001953125f);     // 2^-17, 2^-9
  const long long T = (long long)((unsigned long long)u0 * 0x80000000ull +
                                  ((unsigned long long)u1 * 32768ull + ((unsigned long long)u2 + (kLess + more))));
  const unsigned long long a = (unsigned long long)(T < 0 ? -T : T);
  const float f = __fmaf_rz(__uint2float_rz((uint32_t)(a >> 32)), 4294967296.f, __uint2float_rz((uint32_t)a));
  return ((T < 0 ? -f : f) + low) * scale;
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

// Digits of 128 rows of C = A_{:,K} (C_K = -I), TPR threads per row: image rows
// [Re | Im].  Row i is read from row src[i - 128 mt] when `src` is given.  The
// rows pass through `stage` (128 x kStageRow), brought in by whole 512-byte rows
// (34 us for 384 tiles when every thread read its own row).
constexpr int kStageRow = kNB + 1;
template <int TPR>
__device__ __forceinline__ void pack_c_rows(const double2* __restrict__ A, int np, int k0, int mt, const int* src,
                                            double2* stage, __nv_bfloat16* __restrict__ img, int* __restrict__ cexp,
                                            int* status) {
  constexpr int CNT = kNB / TPR, kWarps = 128 * TPR / 32;
  const int row = threadIdx.x / TPR, part = threadIdx.x % TPR, i = mt * 128 + row;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 8
  for (int r = warp; r < 128; r += kWarps) {
    const int g = mt * 128 + r;
    double2 z = A[box_off(np, src ? src[r] : g, k0 + lane)];
    if (g >= k0 && g < k0 + kNB) z = make_double2(lane == g - k0 ? -1.0 : 0.0, 0.0);
    stage[r * kStageRow + lane] = z;
  }
  __syncthreads();
  double2 z[CNT];
#pragma unroll
  for (int c = 0; c < CNT; ++c) z[c] = stage[row * kStageRow + CNT * part + c];
  unsigned m = 0;
#pragma unroll
  for (int c = 0; c < CNT; ++c) m = max(m, max(mag_hi(z[c].x), mag_hi(z[c].y)));
#pragma unroll
  for (int o = 1; o < TPR; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (m >= 0x7ff00000u && status) atomicCAS(status, 0, DS_SINGULAR);  // not finite
  const int be = row_biased(m);
  if (part == 0) cexp[i] = be - 1022;
#pragma unroll
  for (int im = 0; im < 2; ++im)
#pragma unroll
    for (int g = 0; g < CNT / 8; ++g) {
      long long y[8];
#pragma unroll
      for (int c = 0; c < 8; ++c) y[c] = digit_word(im ? z[8 * g + c].y : z[8 * g + c].x, be);
      const int off = core_off(row, 32 * im + CNT * part + 8 * g);
      put_digits(y, [&](int s, uint4 v) { *reinterpret_cast<uint4*>(img + s * kARow + off) = v; });
    }
}

struct BlockSmem {
  __nv_bfloat16 a[kS * 64 * kK];   // digits of the block: row 2r = [Re | -Im], 2r + 1 = [Im | Re]
  __nv_bfloat16 x[kS * kNB * kK];  // digits of X: row j = [Re X_j | Im X_j], column j over k
  __nv_bfloat16 zero[kNB * kK];    // a zero digit, which opens the sums of order 7
  float2 xt[kNB][kNB], e[kNB][kNB + 2];  // X by columns, the residual by rows
  float2 mult[2][kNB];
  uint64_t bar;
  uint32_t tmem_slot;
  int aexp[kNB], xexp[kNB];
  unsigned amax, emax;
  int abort, bad;
};
// The products read 128 rows of a digit; rows past 64 are the next digit's (the
// last one's: those of X), and their sums are not read.
static_assert(sizeof(BlockSmem::zero) == 256 * 16 && offsetof(BlockSmem, zero) == offsetof(BlockSmem, x) + sizeof(BlockSmem::x),
              "the zero digit follows those of X");
static_assert(128 * kStageRow * sizeof(double2) <= sizeof(BlockSmem), "C rows are staged in the same space");
static_assert(offsetof(BlockSmem, x) == kS * 64 * kK * 2 && kNB * kK * 2 * 2 <= (int)sizeof(BlockSmem::x), "row overrun");

// x as a double, exactly, on the integer units (conversions run on the FP64
// units); zero and subnormals become zero, infinities and NaN large values (the
// caller has checked for them).
__device__ __forceinline__ double widen(float x) {
  const unsigned u = __float_as_uint(x), a = u & 0x7fffffffu;
  return a < 0x00800000u ? 0.0 : __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + (896u << 20))), (int)(u << 29));
}
// x as a float, rounded towards zero, on the integer units; below the range
// zero, above it and for a NaN a NaN.
__device__ __forceinline__ float narrow(double x) {
  const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x);
  const uint32_t e = (hi >> 20) & 0x7ffu;
  uint32_t u = __funnelshift_l(lo, hi, 3) - (896u << 23);
  u = e < 897u ? 0u : e > 896u + 254u ? 0x7fffffffu : u;
  return __uint_as_float((u & 0x7fffffffu) | (hi & 0x80000000u));
}
__device__ __forceinline__ float2 narrow(double2 z) { return make_float2(narrow(z.x), narrow(z.y)); }
__device__ __forceinline__ void cfmaf(float2& acc, float2 a, float2 b) {
  acc.x = fmaf(a.x, b.x, fmaf(-a.y, b.y, acc.x));
  acc.y = fmaf(a.x, b.y, fmaf(a.y, b.x, acc.y));
}

// The inverse of a 32 x 32 FP64 block by 256 threads.  Thread t brings entries
// in[0 .. 3] = (row t / 8, columns 4 (t % 8) ..) and gets out[0 .. 3] = (rows
// 4 (t % 8) .., column t / 8) of the inverse.  False: not found to FP64 accuracy
// this way (the first residual is not small), or perhaps singular by the measure
// of `recip`, a pivot of at most 1e-12, which only the FP64 elimination can tell:
// a small FP32 pivot, or a large inverse.  (The Schur complement of a singular
// matrix is rounding noise, which has an inverse as good as any.  Over contours of
// 26 to 1500 rows with U from 0.3 to 2 the smallest pivot is 0.15, so no such
// block takes the elimination.)
// An FP32 Gauss-Jordan elimination by four warps, then X <- X + X E with the
// residual E = I - A X from the digit products on the tensor cores, with order 7 and
// exact to 2^-60 of the row and column maxima, and the small product X E
// in FP32: E squares from round to round (1e-5, 1e-10 as a rule), and below
// 2^-30 FP32 is enough for the last correction.  Latency bound.  Why: the same block by
// FP64 elimination is 32768 complex multiply-adds on two FP64 units, 33 us at best; the
// kernel with it took 55 us for 64 blocks of matrices of 768 rows, with this 33.
// The residual's last bits decide the accuracy of the whole inversion: with seven orders, 2^-54, G_loc
// erred by 1.2e-15 (N_c = 80) and 7e-15 (220) against long double; with eight by 5e-16
// and 2e-15 (FP64 elimination: 1.1e-15 and 3.7e-15).  The eighth order in the update and
// the R panel changes neither and costs 2 %.
__device__ __forceinline__ bool refined_inverse(BlockSmem& sm, const double2 (&in)[4], double2 (&out)[4],
                                                uint32_t tmem, uint32_t& phase) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int r = t >> 3, c4 = 4 * (t & 7);
  unsigned m = 0;
#pragma unroll
  for (int c = 0; c < 4; ++c) m = max(m, max(mag_hi(in[c].x), mag_hi(in[c].y)));
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (t == 0) {
    sm.amax = 0;
    sm.bad = 0;
  }
  reinterpret_cast<uint4*>(sm.zero)[t] = make_uint4(0, 0, 0, 0);
  __syncthreads();
  if ((t & 7) == 0) atomicMax(&sm.amax, m);
  __syncthreads();
  const unsigned am = sm.amax;
  // FP32 needs the block near one: scaled by 2^-e when its largest entry is not within 2^20
  const int ea = (int)(am >> 20) - 1022, e = ea > 20 || ea < -20 ? ea : 0;
  if (am >= 0x7ff00000u || am < (24u << 20) || ea > 900) return false;
  const double sc = __hiloint2double((1023 - e) << 20, 0);
  // A pivot of at most 2^-10 of the block, or of about 1e-12 before scaling, is left to the FP64 elimination
  // and its test: FP32 cannot tell it from its own rounding.
  const int tiny2 = 2 * (max(ea - 10, -39) - e);
  const float pmin = __int_as_float((127 + max(-126, min(127, tiny2))) << 23);
  const int be = row_biased(m);
  {
    long long y[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      y[c] = digit_word(in[c].x, be);
      y[4 + c] = digit_word(in[c].y, be);
      sm.xt[c4 + c][r] = narrow(e == 0 ? in[c] : make_double2(in[c].x * sc, in[c].y * sc));
    }
    if ((t & 7) == 0) sm.aexp[r] = be - 1022 - e;
    const int o_re = core_off(2 * r, c4), o_im = core_off(2 * r, 32 + c4);
    put_digits(y, [&](int s, uint4 w) {
      __nv_bfloat16* d = sm.a + s * 64 * kK;
      const uint4 n = neg_bf16(w);
      *reinterpret_cast<uint2*>(d + o_re) = make_uint2(w.x, w.y);
      *reinterpret_cast<uint2*>(d + o_im) = make_uint2(n.z, n.w);
      *reinterpret_cast<uint2*>(d + o_re + 8) = make_uint2(w.z, w.w);
      *reinterpret_cast<uint2*>(d + o_im + 8) = make_uint2(w.x, w.y);
    });
  }
  __syncthreads();
  if (warp < 4) {
    // lane = row, eight columns per warp; the step's column's warp sends every row's multiplier
    float2 v[8];
#pragma unroll
    for (int c = 0; c < 8; ++c) v[c] = sm.xt[8 * warp + c][lane];
    bool good = true;
#pragma unroll 1
    for (int kw = 0; kw < 4; ++kw)
#pragma unroll
      for (int kc = 0; kc < 8; ++kc) {
        const int k = 8 * kw + kc;
        float2 p[8];  // this warp's part of the pivot row
#pragma unroll
        for (int c = 0; c < 8; ++c)
          p[c] = make_float2(__shfl_sync(0xffffffffu, v[c].x, k), __shfl_sync(0xffffffffu, v[c].y, k));
        if (warp == kw) {
          const float pm = p[kc].x * p[kc].x + p[kc].y * p[kc].y;
          good = good && pm > pmin;
          float rm;
          asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rm) : "f"(pm));
          const float2 pinv = make_float2(p[kc].x * rm, -p[kc].y * rm);
          // row k: -1 / pivot, on a row taken as zero; the others: their entry over the pivot
          sm.mult[kc & 1][lane] = lane == k ? make_float2(-pinv.x, -pinv.y)
                                            : make_float2(v[kc].x * pinv.x - v[kc].y * pinv.y,
                                                          v[kc].x * pinv.y + v[kc].y * pinv.x);
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const float2 f = sm.mult[kc & 1][lane], nf = make_float2(-f.x, -f.y);
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          if (lane == k) v[c] = make_float2(0.f, 0.f);
          cfmaf(v[c], nf, p[c]);
        }
        if (warp == kw) v[kc] = nf;
      }
#pragma unroll
    for (int c = 0; c < 8; ++c) sm.xt[8 * warp + c][lane] = v[c];
    if (!good) sm.bad = 1;
  }
  __syncthreads();
  // from here on thread t holds rows c4 .. c4 + 3 of column r of X
  const int j = r;
#pragma unroll
  for (int c = 0; c < 4; ++c) out[c] = make_double2(widen(sm.xt[j][c4 + c].x), widen(sm.xt[j][c4 + c].y));
  if (sm.bad) return false;
  for (int round = 0; round < 4; ++round) {
    unsigned mx = 0;
#pragma unroll
    for (int c = 0; c < 4; ++c) mx = max(mx, max(mag_hi(out[c].x), mag_hi(out[c].y)));
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    const int bx = row_biased(mx);
    if ((t & 7) == 0) sm.xexp[j] = bx - 1022 - e > 39 ? 1000 : bx - 1022;  // about 1e12 and more: as a lost column
    if (t == 0) sm.emax = 0;
    long long y[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      y[c] = digit_word(out[c].x, bx);
      y[4 + c] = digit_word(out[c].y, bx);
    }
    const int o_re = core_off(j, c4), o_im = core_off(j, 32 + c4);
    put_digits(y, [&](int s, uint4 w) {
      __nv_bfloat16* d = sm.x + s * kNB * kK;
      *reinterpret_cast<uint2*>(d + o_re) = make_uint2(w.x, w.y);
      *reinterpret_cast<uint2*>(d + o_im) = make_uint2(w.z, w.w);
    });
    fence_proxy_async();
    __syncthreads();
    if (t == 0) {
      tc_fence_after();
#pragma unroll
      for (int a = 0; a < kS; ++a)
#pragma unroll
        for (int kk = 0; kk < kK / 16; ++kk)
          mma_bf16(tmem + (uint32_t)(a * kNB), smem_desc(smem_u32(sm.a + a * 64 * kK) + kk * 256, 128, 1024),
                   smem_desc(smem_u32(sm.x) + kk * 256, 128, 1024),
                   idesc_bf16(128, (a == 0 && kk > 0 ? kS : kO - a) * kNB),
                   (a > 0 || kk > 0) ? 1u : 0u);
      mma_commit(&sm.bar);
    }
    volatile int* abort_flag = &sm.abort;
    bool ok = mbar_wait(&sm.bar, phase, abort_flag);
    if (!ok) drain_wait(&sm.bar, phase);
    phase ^= 1u;
    if (!__syncthreads_and(ok)) return false;
    tc_fence_after();
    if ((warp & 3) < 2) {  // lanes 2 r, 2 r + 1 of the first two quarters hold Re, Im of row r; two warps halve the columns
      const int row = (warp & 3) * 16 + (lane >> 1), part = lane & 1, j0 = 16 * (warp >> 2);
      float big = 0.f;
#pragma unroll 1
      for (int g = 0; g < 16; g += 8) {
        float c[kO][8];
#pragma unroll
        for (int o = 0; o < kO; ++o)
          tmem_ld8(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(o * kNB + j0 + g), c[o]);
        tmem_wait_ld();
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          // A X - I in units of 2^(ex - 53), the one taken off before any rounding
          const int col = j0 + g + u, ex = sm.aexp[row] + sm.xexp[col];
          const bool one = row == col && part == 0;
          if (one && (ex < -8 || ex > 50)) big = 1e30f;  // not an inverse: a column of X or a row of A is lost
          const float f = -orders_to_float(c[0][u], c[1][u], c[2][u], c[3][u], c[4][u], c[5][u], c[6][u], c[7][u],
                                           one ? 0ull - (1ull << ((53 - ex) & 63)) : 0ull,
                                           __int_as_float((127 - 53 + max(min(ex, 100), -60)) << 23));
          big = fmaxf(big, fabsf(f));
          (&sm.e[row][col].x)[part] = f;
        }
      }
      tc_fence_before();
      const unsigned wb = __reduce_max_sync(0xffffffffu, __float_as_uint(big));
      if (lane == 0) atomicMax(&sm.emax, wb);
    }
    __syncthreads();
    const float emax = __uint_as_float(sm.emax);
    if (!(emax < 0.125f)) return false;
    // X += X E: lane = row of the product, four columns per warp (X by columns and
    // broadcasts of E: four shared-memory wavefronts per l), then back to this thread's entries
    float2 acc[4] = {};
#pragma unroll 8
    for (int l = 0; l < kNB; ++l) {
      const float2 x = sm.xt[l][lane];
      const float4 e01 = *reinterpret_cast<const float4*>(&sm.e[l][4 * warp]);
      const float4 e23 = *reinterpret_cast<const float4*>(&sm.e[l][4 * warp + 2]);
      cfmaf(acc[0], x, make_float2(e01.x, e01.y));
      cfmaf(acc[1], x, make_float2(e01.z, e01.w));
      cfmaf(acc[2], x, make_float2(e23.x, e23.y));
      cfmaf(acc[3], x, make_float2(e23.z, e23.w));
    }
    __syncthreads();  // every thread has read xt and e
#pragma unroll
    for (int c = 0; c < 4; ++c) sm.xt[4 * warp + c][lane] = acc[c];
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float2 d = sm.xt[j][c4 + c];
      out[c].x += widen(d.x);
      out[c].y += widen(d.y);
    }
    const bool last = emax < 9.3e-10f;  // 2^-30: what is left is E^2 and the product's FP32 rounding
    if (last) {
      if (e != 0) {
#pragma unroll
        for (int c = 0; c < 4; ++c) out[c] = make_double2(out[c].x * sc, out[c].y * sc);
      }
      return true;
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) sm.xt[j][c4 + c] = narrow(out[c]);
  }
  return false;
}

// P = inv of a 32 x 32 block by FP64 elimination, 256 threads, a warp per four
// rows (v), lane = column.  Step k: the pivot row, divided by its pivot (its own
// entry replaced by the pivot's inverse), is in shared memory (two buffers, one
// barrier per step); every other row subtracts its entry of column k times it,
// that entry counted as zero before.  The warp of the next pivot row takes that
// row first and publishes it.  FP64 bound: 32 rows x 4 FMAs x 16 cycles per step.
__device__ __forceinline__ void fp64_inverse(double2 (&v)[4], double2 (&rowb)[2][32], int* status) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
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
}

// Matrix b's P (rows in shared memory) to Pbuf, and the digits of its 64 real
// rows, eight threads per row r, four entries each: row 2r = [Re P_r | -Im P_r],
// row 2r + 1 = [Im P_r | Re P_r].
__device__ __forceinline__ void write_p(const double2 (*prow)[kNB + 1], int b, double2* __restrict__ Pbuf,
                                        __nv_bfloat16* __restrict__ pimg, int* __restrict__ pexp, int* status) {
  const int t = threadIdx.x;
  const int r = t >> 3, c4 = 4 * (t & 7);
  double2 p[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    p[c] = prow[r][c4 + c];
    Pbuf[(size_t)b * kNB * kNB + r * kNB + c4 + c] = p[c];
  }
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
}

// P = inv of the block with entries entry(row, column), by 256 threads, and its
// digits; all of the CTA's threads, with the shared memory to themselves.
template <class Entry>
__device__ __forceinline__ void invert_block(BlockSmem& sm, Entry&& entry, int b, double2* __restrict__ Pbuf,
                                             __nv_bfloat16* __restrict__ pimg, int* __restrict__ pexp, int* status) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int r = t >> 3, c4 = 4 * (t & 7);
  double2 in[4], out[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) in[c] = entry(r, c4 + c);
  if (t == 0) {
    mbar_init(&sm.bar, 1);
    sm.abort = 0;
    fence_barrier_init();
  }
  if (warp == 0) tmem_alloc(&sm.tmem_slot, 256);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sm.tmem_slot;
  uint32_t phase = 0;
  const bool found = refined_inverse(sm, in, out, tmem, phase);
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, 256);
  }
  if (t == 0 && sm.abort && status) atomicCAS(status, 0, DS_TIMEOUT);
  // P by rows through shared memory (over the digits, which nobody reads any more)
  double2 (*prow)[kNB + 1] = reinterpret_cast<double2 (*)[kNB + 1]>(sm.a);
  if (found) {
#pragma unroll
    for (int c = 0; c < 4; ++c) prow[c4 + c][r] = out[c];
  } else {
    double2 v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = entry(4 * warp + q, lane);
    fp64_inverse(v, *reinterpret_cast<double2 (*)[2][32]>(sm.x), status);
#pragma unroll
    for (int q = 0; q < 4; ++q) prow[4 * warp + q][lane] = v[q];
  }
  __syncthreads();
  write_p(prow, b, Pbuf, pimg, pexp, status);
}

// CTAs 0 .. nb-1: P = inv(A_KK) of matrix b and its digits.
// CTAs nb ..: digits of 128 rows of C, two threads per row; this work hides
// behind the pivot blocks' latency.
__global__ void __launch_bounds__(256, 2)
    gj64_pivot_kernel(const double2* __restrict__ A, int np, int mtiles, int k0, int nb, double2* __restrict__ Pbuf,
                      __nv_bfloat16* __restrict__ pimg, int* __restrict__ pexp, __nv_bfloat16* __restrict__ cimg,
                      int* __restrict__ cexp, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  if ((int)blockIdx.x < nb) {
    const double2* a = A + (size_t)blockIdx.x * np * np;
    invert_block(*reinterpret_cast<BlockSmem*>(smem_raw), [&](int r, int c) { return a[box_off(np, k0 + r, k0 + c)]; },
                 blockIdx.x, Pbuf, pimg, pexp, status);
    return;
  }
  const int u = blockIdx.x - nb, b = u / mtiles, mt = u % mtiles;
  pack_c_rows<2>(A + (size_t)b * np * np, np, k0, mt, nullptr, reinterpret_cast<double2*>(smem_raw),
                 cimg + (size_t)u * kATile, cexp + (size_t)b * np,
                 status);
}

// ------------------------------------------------------------------ R panel

// The row exchanges of one pivoted step: the row chosen for each place of block
// K, and the block's rows that move out to the chosen rows' places.
struct RowSwaps {
  int win[kNB];
  int moved, to[kNB], from[kNB];
};

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
// One CTA per SM, its phases one after the other: latency bound, hence 16 warps
// (47 us for 64 matrices of 768 rows, 32 us for 64 of 256).
// With `sw` (one matrix, pivoted): row k0 + r of A_K is row sw->win[r]; the rows
// that leave block K for the winners' places are copied there, each CTA its own
// columns; and CTAs mtiles .. 2 mtiles - 1 cut C into digits with the rows so
// moved.  No CTA writes what another reads: the copies go to the winners' rows,
// whose only readers are the CTA of the same columns, before its copies.
__global__ void __launch_bounds__(512, 1)
    gj64_rpanel_kernel(double2* A, int np, int mtiles, int k0, const double2* __restrict__ Pbuf,
                       const __nv_bfloat16* __restrict__ pimg, const int* __restrict__ pexp,
                       __nv_bfloat16* __restrict__ rimg, int* __restrict__ rexp, const RowSwaps* __restrict__ sw,
                       __nv_bfloat16* __restrict__ cimg, int* __restrict__ cexp, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  if ((int)blockIdx.x >= mtiles) {
    __shared__ int src[128];
    const int mt = blockIdx.x - mtiles, t = threadIdx.x;
    if (t < 128) src[t] = mt * 128 + t;
    __syncthreads();
    if (t < sw->moved && sw->to[t] / 128 == mt) src[sw->to[t] % 128] = sw->from[t];
    __syncthreads();
    pack_c_rows<4>(A, np, k0, mt, src, reinterpret_cast<double2*>(smem_raw), cimg + (size_t)mt * kATile, cexp, status);
    return;
  }
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
  double2* mat = A + (size_t)b * np * np;
#pragma unroll
  for (int c = 0; c < 8; ++c) z[c] = mat[box_off(np, sw ? sw->win[8 * h + c] : k0 + 8 * h + c, j)];
  tc_fence_before();
  __syncthreads();  // barriers, colmax, TMEM address; every row of A_K is read
  tc_fence_after();
  if (sw)
    for (int e = h; e < sw->moved; e += 4) mat[box_off(np, sw->to[e], j)] = mat[box_off(np, sw->from[e], j)];
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
// 2-9 drain: a thread has one row and 8 complex columns, a warp one 4 KB box of 32
// rows x 128 bytes (contiguous in A), which is added to A at L2 by a bulk FP64
// reduction (rows and columns of block K: stored).  Column tiles at or past `jskip`
// move up by `nskip` (a window that another kernel updates).
// What bounds it: HBM.  A passes through L2 once per step, read and written by the
// additions: 64 matrices of 700 rows (np = 768) in 222 us with 1.38 GB of DRAM traffic
// (counters), 6.2 TB/s, 0.91 of the copy rate.  Close behind: a tile's products take 2305 cycles
// of 3600 (an MMA of 128 rows and K = 16 takes max(72, N / 2)), the epilogue about 1700
// issue cycles.  Left out one at a time (of 238 us then): the additions 210 us, the epilogue's arithmetic 238,
// the loads of R 220, the additions and the products' width 208.  Boxes of rows past n
// are not touched: N_c = 700 7.84 -> 7.66 ms, 1500 42.1 -> 41.5 (around the epilogue's
// arithmetic too, the same test made it 10 % slower).  Measured before: old values loaded
// by TMA in 64-byte rows two boxes ahead, subtracted and stored, 292 us (the shared
// memory left for boxes does not cover the latency); half of the boxes each way, 274 us;
// every other tile of six warps loaded in 128-byte rows one tile ahead, 359 us; the
// additions as 2-D boxes of a row-major A, 243 us.  FP64 units: 20.6 ms for all 47 steps of a
// matrix of 1500 rows; here 0.85 ms, the panels included.
__global__ void __launch_bounds__(64 + 32 * kEpiW, 1)
    gj64_update_kernel(double2* __restrict__ A, int n, int np, int mtiles, int ntn, int total, int k0,
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
    // exponents of a tile's row and eight columns, fetched a tile ahead (N_c = 700, 64 points
    // 7.68 -> 7.51 ms, 1500 unchanged)
    int4 ej[2];
    int ei = 0;
    auto exponents = [&](const Pos& p) {
      const int* r = rexp + (size_t)p.b * np + col_tile(p.jn) * kTn + c0;
      ej[0] = *reinterpret_cast<const int4*>(r);
      ej[1] = *reinterpret_cast<const int4*>(r + 4);
      ei = cexp[(size_t)p.b * np + p.mt * 128 + quarter * 32 + lane] + 1023 - 53;
    };
    if (lo < hi) exponents(cur);
    bool ok = true;
    for (int tile = lo, it = 0; tile < hi && ok; ++tile, ++it) {
      const int jt = col_tile(cur.jn), s = it & 1;
      const int b = cur.b, i = cur.mt * 128 + quarter * 32 + lane;
      const bool ik = i >= k0 && i < k0 + kNB;  // the same for the whole warp
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
      if (lane == 0) {
        mbar_arrive(&bars.d_empty[s]);
        bulk_wait_read_n<0>();  // the last tile's box has been read
      }
      __syncwarp();
      const int j = jt * kTn + c0;
      const int eb8[8] = {ei + ej[0].x, ei + ej[0].y, ei + ej[0].z, ei + ej[0].w,
                          ei + ej[1].x, ei + ej[1].y, ei + ej[1].z, ei + ej[1].w};
      step(cur);
      if (tile + 1 < hi) exponents(cur);
#pragma unroll
      for (int hb = 0; hb < 2; ++hb) {
        const float(&c)[kS][8] = acc[hb];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int eb = eb8[4 * hb + q];
          const double dx = orders_to_double(c[0][2 * q], c[1][2 * q], c[2][2 * q], c[3][2 * q], c[4][2 * q],
                                             c[5][2 * q], c[6][2 * q], eb);
          const double dy = orders_to_double(c[0][2 * q + 1], c[1][2 * q + 1], c[2][2 * q + 1], c[3][2 * q + 1],
                                             c[4][2 * q + 1], c[5][2 * q + 1], c[6][2 * q + 1], eb);
          *reinterpret_cast<double2*>(box + lane * 128 + (((4 * hb + q) ^ (lane & 7)) << 4)) = make_double2(-dx, -dy);
        }
      }
      fence_proxy_async();
      __syncwarp();
      if (lane == 0 && i < n) {  // a box of rows past n stays as it is (zero times anything)
        double2* dst = A + (size_t)b * np * np + box_off(np, i, j & ~7);  // lane 0: row 0 of the box
        if (ik || (j >= k0 && j < k0 + kNB)) bulk_store(dst, box, kBoxBytes);  // block K: nothing to add to
        else bulk_add_f64(dst, box, kBoxBytes);
        bulk_commit();
      }
      __syncwarp();
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
  int sms = 0;
  int rc = device_sm_count(&sms);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_pivot_kernel), (int)sizeof(BlockSmem));
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_rpanel_kernel), RSmem::kBytes);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_update_kernel), USmem::kBytes);
  if (rc) return rc;
  const int mtiles = np / 128, ntn = ceil_div(n, kTn), total = nb * mtiles * ntn;
  for (int k0 = 0; k0 < n; k0 += kNB) {
    gj64_pivot_kernel<<<nb + nb * mtiles, 256, sizeof(BlockSmem), st>>>(A, np, mtiles, k0, nb, pbuf, pimg, pexp, cimg,
                                                          cexp, status);
    NED_LAUNCH_CHECK("gj64_pivot_kernel");
    gj64_rpanel_kernel<<<dim3(mtiles, nb), 512, RSmem::kBytes, st>>>(A, np, mtiles, k0, pbuf, pimg, pexp, rimg, rexp,
                                                                     nullptr, nullptr, nullptr, status);
    NED_LAUNCH_CHECK("gj64_rpanel_kernel");
    const int slot = instr_begin(st);
    gj64_update_kernel<<<total < sms ? total : sms, 64 + 32 * kEpiW, USmem::kBytes, st>>>(
        A, n, np, mtiles, ntn, total, k0, ntn, 0, cimg, cexp, rimg, rexp, status);
    NED_LAUNCH_CHECK("gj64_update_kernel");
    const int live = n - k0 < kNB ? n - k0 : kNB;
    instr_end(slot, st, 8.0 * (double)n * n * live * nb, 2.0 * sizeof(double2) * (double)n * n * nb);
  }
  return NEDMFT_OK;
}

// ------------------------------------------------------------------ pivoted inversion of one matrix

namespace {

constexpr int kPanThreads = 256;
constexpr int kPanCand = 256;  // candidate rows of a CTA
constexpr int kPanCtas = 8;    // most CTAs of a cluster
constexpr int kPanRows = kPanCand * kPanCtas;

constexpr int kStagePitch = kNB + 1;  // staged candidate rows: conflict-free with a lane per row
struct PanSmem {
  float4 prow[2][kNB / 2];  // the pivot row, from the step's column on (by step parity)
  int4 key[2];              // the four warps' largest |entry|^2 as ordered bits
  int win[kNB];
  int cand[kPanCand];
};

// Partial pivoting in FP32 on a CTA's candidate rows sm.cand (-1: none) over the
// 32 columns from k0 on; the rows chosen, in order, to sm.win.  The rows come in
// coalesced, through `stage` (256 x kStagePitch float2); then four warps keep two
// rows per lane in registers.  Per column: a warp maximum, one over the four
// warps, the chosen row to shared memory, and every lane eliminates its rows,
// writing the result one register down, so that the column in hand is always
// register 0 and the loop needs no unrolling.  A step is latency and the pivot
// row's broadcast (256 bytes per lane, hence two rows per lane): 720 cycles on
// average; 1230 with a row per thread in eight warps and every warp's best row
// published before one barrier; 1830 with one exchange per column through a
// cluster of eight CTAs, which saves the second round (the same 9.5 ms per
// impurity step at N_c = 1500, but 542 us against 470 at N_c = 80).
__device__ __forceinline__ void choose_rows(PanSmem& sm, float2* stage, const double2* __restrict__ A, int np, int n,
                                            int k0) {
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int ncol = min(kNB, n - k0);
#pragma unroll 8
  for (int r = warp; r < kPanCand; r += kPanThreads / 32) {
    const int row = sm.cand[r];
    const float2 f = narrow(A[box_off(np, max(row, k0), k0 + lane)]);  // loaded either way: the loads overlap
    stage[r * kStagePitch + lane] = row >= 0 && lane < ncol ? f : make_float2(0.f, 0.f);
  }
  if (t < kNB) sm.win[t] = -1;
  __syncthreads();
  if (warp < 4) {
    float2 v[2][kNB];
    bool live[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = 64 * warp + 32 * h + lane;
      live[h] = sm.cand[r] >= 0;
#pragma unroll
      for (int e = 0; e < kNB; ++e) v[h][e] = stage[r * kStagePitch + e];
    }
    // columns past the panel's shift in as zeros: after 16 and 24 steps half and a quarter of the registers are left
    auto steps = [&](auto width, int j0, int j1) {
      constexpr int W = decltype(width)::value;
#pragma unroll 1
      for (int j = j0; j < j1; ++j) {
        const int sb = j & 1;
        // |entry|^2 as ordered bits, -1 below every magnitude; a NaN is never chosen
        const float m0 = v[0][0].x * v[0][0].x + v[0][0].y * v[0][0].y;
        const float m1 = v[1][0].x * v[1][0].x + v[1][0].y * v[1][0].y;
        const int k_0 = live[0] && m0 >= 0.f ? __float_as_int(m0) : -1;
        const int k_1 = live[1] && m1 >= 0.f ? __float_as_int(m1) : -1;
        const bool second = k_1 > k_0;
        const int key = second ? k_1 : k_0;
        const int top = __reduce_max_sync(0xffffffffu, key);
        const int src = __ffs(__ballot_sync(0xffffffffu, key == top)) - 1;
        if (lane == src) (&sm.key[sb].x)[warp] = top;
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const int4 y = sm.key[sb];
        const int best = max(max(y.x, y.y), max(y.z, y.w));
        const int wtop = best == y.x ? 0 : best == y.y ? 1 : best == y.z ? 2 : 3;
        if (warp == wtop && lane == src) {
          if (second) {
#pragma unroll
            for (int e = 0; e < W / 2; ++e)
              sm.prow[sb][e] = make_float4(v[1][2 * e].x, v[1][2 * e].y, v[1][2 * e + 1].x, v[1][2 * e + 1].y);
            live[1] = false;
          } else {
#pragma unroll
            for (int e = 0; e < W / 2; ++e)
              sm.prow[sb][e] = make_float4(v[0][2 * e].x, v[0][2 * e].y, v[0][2 * e + 1].x, v[0][2 * e + 1].y);
            live[0] = false;
          }
          if (best >= 0) sm.win[j] = sm.cand[64 * warp + (second ? 32 : 0) + lane];  // else none left, or none finite
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        const float4* pr = sm.prow[sb];
        const float4 p0 = pr[0];
        const float pm = p0.x * p0.x + p0.y * p0.y;
        float rm;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(rm) : "f"(pm));
        rm = pm > 1e-37f ? rm : 0.f;
        float2 f[2];
#pragma unroll
        for (int h = 0; h < 2; ++h)
          f[h] = make_float2((v[h][0].x * p0.x + v[h][0].y * p0.y) * rm, (v[h][0].y * p0.x - v[h][0].x * p0.y) * rm);
#pragma unroll
        for (int e = 0; e < W / 2; ++e) {
          const float4 z = e == 0 ? p0 : pr[e];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (e > 0) v[h][2 * e - 1] = make_float2(fmaf(-f[h].x, z.x, fmaf(f[h].y, z.y, v[h][2 * e].x)),
                                                     fmaf(-f[h].x, z.y, fmaf(-f[h].y, z.x, v[h][2 * e].y)));
            v[h][2 * e] = make_float2(fmaf(-f[h].x, z.z, fmaf(f[h].y, z.w, v[h][2 * e + 1].x)),
                                      fmaf(-f[h].x, z.w, fmaf(-f[h].y, z.z, v[h][2 * e + 1].y)));
          }
        }
        v[0][W - 1] = v[1][W - 1] = make_float2(0.f, 0.f);
      }
    };
    steps(std::integral_constant<int, 32>{}, 0, min(ncol, 16));
    steps(std::integral_constant<int, 16>{}, 16, min(ncol, 24));
    steps(std::integral_constant<int, 8>{}, 24, ncol);
  }
  __syncthreads();
}

// Pivot choice for the 32 columns from k0 on and, in the last round, the block's
// inverse.  A tournament: each CTA of a cluster chooses 32 of its 256 candidate
// rows (rows k0 + i, or in[i]), then the cluster's first CTA 32 of those.  Last
// round: P = inv of the chosen rows' block and its digits, the row exchanges, the
// row permutation.  Latency bound throughout.
__global__ void __launch_bounds__(kPanThreads, 1)
    gj64_panel_kernel(const double2* __restrict__ A, int np, int n, int k0, const int* __restrict__ in, int count,
                      int* __restrict__ out, int last, double2* __restrict__ Pbuf, __nv_bfloat16* __restrict__ pimg,
                      int* __restrict__ pexp, RowSwaps* __restrict__ sw, int* __restrict__ rowperm, int* status) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  BlockSmem& blk = *reinterpret_cast<BlockSmem*>(smem_raw);
  PanSmem& sm = *reinterpret_cast<PanSmem*>(smem_raw + (sizeof(BlockSmem) + 127) / 128 * 128);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  uint32_t nq;
  asm volatile("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(nq));
  const int q = (int)cluster_ctarank();
  float2* stage = reinterpret_cast<float2*>(smem_raw);
  const int i = blockIdx.x * kPanCand + t;
  sm.cand[t] = i < count ? (in ? in[i] : k0 + i) : -1;
  __syncthreads();
  choose_rows(sm, stage, A, np, n, k0);
  if (nq > 1) {
    cluster_sync();  // the first CTA has read its own candidates
    if (t < kNB)
      asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(cluster_addr(&sm.cand[q * kNB + t], 0)), "r"(sm.win[t])
                   : "memory");
    cluster_sync();
    if (q > 0) return;
    if (t >= (int)nq * kNB) sm.cand[t] = -1;
    __syncthreads();
    choose_rows(sm, stage, A, np, n, k0);
  }
  if (!last) {
    if (t < kNB) out[(blockIdx.x / nq) * kNB + t] = sm.win[t];
    return;
  }
  invert_block(blk, [&](int r, int c) { return A[box_off(np, sm.win[r] >= 0 ? sm.win[r] : k0 + r, k0 + c)]; }, 0, Pbuf,
               pimg, pexp, status);
  if (warp == 0) {
    // place k0 + lane takes row w; a winner from outside the block leaves its
    // place to a row of the block that was not chosen (the t-th such place gets
    // the t-th such row)
    const int w = sm.win[lane] >= 0 ? sm.win[lane] : k0 + lane;
    const bool inside = w >= k0 && w < k0 + kNB;
    if (sm.win[lane] < 0 && k0 + lane < n && status) atomicCAS(status, 0, DS_SINGULAR);  // too few candidates
    const unsigned chosen = __reduce_or_sync(0xffffffffu, inside ? 1u << (w - k0) : 0u);
    const unsigned outs = __ballot_sync(0xffffffffu, !inside);
    const int at = __popc(outs & ((1u << lane) - 1u));
    unsigned left = ~chosen;
    for (int u = 0; u < at; ++u) left &= left - 1;  // drop the lowest
    const int from = k0 + __ffs(left) - 1;
    const int pw = rowperm[w], pf = inside ? 0 : rowperm[from];
    __syncwarp();
    rowperm[k0 + lane] = pw;
    sw->win[lane] = w;
    if (!inside) {
      rowperm[w] = pf;
      sw->to[at] = w;
      sw->from[at] = from;
    }
    if (lane == 0) sw->moved = __popc(outs);
  }
}

static_assert(kPanCand * kStagePitch * sizeof(float2) <= sizeof(BlockSmem), "candidate rows are staged in the block's space");
constexpr int kPanSmem = (int)((sizeof(BlockSmem) + 127) / 128 * 128 + sizeof(PanSmem));

int launch_panel(const double2* A, int np, int n, int k0, const int* in, int count, int* out, bool last, double2* pbuf,
                 __nv_bfloat16* pimg, int* pexp, RowSwaps* sw, int* rowperm, int* status, cudaStream_t s) {
  // 256 candidate rows per CTA: clusters of 1, 2, 4 or 8 CTAs, the fewest that hold them
  int ctas = 1;
  while (ctas < kPanCtas && ctas * kPanCand < count) ctas *= 2;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(ceil_div(count, ctas * kPanCand) * ctas);
  cfg.blockDim = dim3(kPanThreads);
  cfg.dynamicSmemBytes = kPanSmem;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = ctas;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  NED_CUDA(cudaLaunchKernelEx(&cfg, gj64_panel_kernel, A, np, n, k0, in, count, out, (int)last, pbuf, pimg, pexp, sw,
                              rowperm, status));
  instr_count();
  return NEDMFT_OK;
}

// The inversion works on A 2^-e, e the exponent of max |Re|, |Im| over A
// (exact scaling): its pivot thresholds are then relative and the FP32 pivot
// choice stays in range.  amax holds the bits of that maximum (non-negative
// doubles order like their bit patterns), set by amax_kernel after a clear.
__device__ __forceinline__ int amax_exponent(const unsigned long long* amax) {
  const double m = __longlong_as_double((long long)*amax);
  int e = 0;
  if (m > 0.0 && m <= 1.7976931348623157e308) frexp(m, &e);
  return e;
}

__global__ void amax_kernel(const double2* __restrict__ a, size_t total, unsigned long long* __restrict__ amax) {
  double m = 0.0;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const double2 z = a[e];
    m = fmax(m, fmax(fabs(z.x), fabs(z.y)));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) atomicMax(amax, (unsigned long long)__double_as_longlong(m));
}

// The scaled copy, padded with the identity, and the identity row permutation.
__global__ void pad_identity_kernel(const double2* __restrict__ a, int n, double2* __restrict__ ap, int np,
                                    const unsigned long long* __restrict__ amax, int* __restrict__ rowperm) {
  const int sh = -amax_exponent(amax);
  const int i = blockIdx.x;
  for (int j = blockIdx.y * blockDim.x + threadIdx.x; j < np; j += gridDim.y * blockDim.x) {
    double2 v = make_double2(i == j ? 1.0 : 0.0, 0.0);
    if (i < n && j < n) {
      const double2 z = a[(size_t)i * n + j];
      v = make_double2(scalbn(z.x, sh), scalbn(z.y, sh));
    }
    ap[box_off(np, i, j)] = v;
    if (i == 0) rowperm[j] = j;
  }
}

// y = the inverse of A from x = (P A 2^-e)^-1: column c of x is column
// rowperm[c] of A^-1, and inv(A 2^-e) = 2^e inv(A)
__global__ void unpermute_kernel(const double2* __restrict__ x, int np, int n, const int* __restrict__ rowperm,
                                 double2* __restrict__ y, const unsigned long long* __restrict__ amax) {
  const int sh = -amax_exponent(amax);
  const int i = blockIdx.x;
  for (int c = blockIdx.y * blockDim.x + threadIdx.x; c < n; c += gridDim.y * blockDim.x) {
    const double2 z = x[box_off(np, i, c)];
    y[(size_t)i * n + rowperm[c]] = make_double2(scalbn(z.x, sh), scalbn(z.y, sh));
  }
}

// Second stream (highest priority) and two events per device and host
// thread for the look-ahead below, created on first use and kept.
struct LookAhead {
  cudaStream_t side = nullptr;
  cudaEvent_t panel = nullptr, chain = nullptr;
};

int look_ahead(LookAhead** out) {
  constexpr int kMaxDev = 64;
  thread_local LookAhead la[kMaxDev];
  int dev = 0;
  NED_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDev) return set_error(NEDMFT_ECUDA, "pivot_inverse: device %d out of range", dev);
  LookAhead& l = la[dev];
  if (!l.side) {
    int lo = 0, hi = 0;
    NED_CUDA(cudaDeviceGetStreamPriorityRange(&lo, &hi));
    NED_CUDA(cudaEventCreateWithFlags(&l.panel, cudaEventDisableTiming));
    NED_CUDA(cudaEventCreateWithFlags(&l.chain, cudaEventDisableTiming));
    NED_CUDA(cudaStreamCreateWithPriority(&l.side, cudaStreamNonBlocking, hi));
  }
  *out = &l;
  return NEDMFT_OK;
}

struct PivLayout {
  size_t a, gj, cand, sw, perm, amax, total;
};
PivLayout piv_layout(int n) {
  PivLayout L;
  const int np = ceil_div(n, 128) * 128;
  L.a = align256(sizeof(double2) * (size_t)np * np);
  L.gj = gj64_layout(np, 1).total;
  L.cand = align256(sizeof(int) * (size_t)ceil_div(n, kPanRows) * kNB);
  L.sw = align256(sizeof(RowSwaps));
  L.perm = align256(sizeof(int) * (size_t)np);
  L.amax = align256(8);
  L.total = L.a + L.gj + 2 * L.cand + L.sw + L.perm + L.amax;
  return L;
}

}  // namespace

size_t pivot_inverse_workspace(int n) { return piv_layout(n).total; }

// Creates this host thread's look-ahead stream and events on the current
// device and sets the kernels' shared-memory limits: for callers that are
// about to capture pivot_inverse into a CUDA graph.
int pivot_inverse_prepare() {
  LookAhead* la = nullptr;
  int rc = look_ahead(&la), sms = 0;
  if (!rc) rc = device_sm_count(&sms);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_panel_kernel), kPanSmem);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_rpanel_kernel), RSmem::kBytes);
  if (!rc) rc = ensure_dyn_smem(reinterpret_cast<const void*>(gj64_update_kernel), USmem::kBytes);
  return rc;
}

// In-place inverse of one n x n matrix with partial pivoting (the impurity
// step), blocked Gauss-Jordan in steps of 32 columns.  Every step's pivot choice
// and pivot-block inverse depend only on its 32 panel columns, so they run one
// step ahead on the second stream: there the update kernel brings the next
// panel's two column tiles up to date, then the panel kernel of step k + 1 runs,
// while step k updates the rest of the matrix on the caller's stream.  The R
// panel of step k + 1 waits for both and moves the rows.  The serial path of a
// step is R panel, window, pivot choice and block inverse.
int pivot_inverse(double2* a, int n, void* ws, cudaStream_t st, int* status) {
  const int np = ceil_div(n, 128) * 128;
  const PivLayout L = piv_layout(n);
  const Gj64Layout G = gj64_layout(np, 1);
  char* p = static_cast<char*>(ws);
  double2* ap = reinterpret_cast<double2*>(p); p += L.a;
  double2* pbuf = reinterpret_cast<double2*>(p); p += G.p;
  __nv_bfloat16* pimg = reinterpret_cast<__nv_bfloat16*>(p); p += G.pi;
  int* pexp = reinterpret_cast<int*>(p); p += G.pe;
  __nv_bfloat16* cimg = reinterpret_cast<__nv_bfloat16*>(p); p += G.c;
  __nv_bfloat16* rimg = reinterpret_cast<__nv_bfloat16*>(p); p += G.r;
  int* cexp = reinterpret_cast<int*>(p); p += G.ce;
  int* rexp = reinterpret_cast<int*>(p); p += G.re;
  int* cand[2];
  cand[0] = reinterpret_cast<int*>(p); p += L.cand;
  cand[1] = reinterpret_cast<int*>(p); p += L.cand;
  RowSwaps* sw = reinterpret_cast<RowSwaps*>(p); p += L.sw;
  int* rowperm = reinterpret_cast<int*>(p); p += L.perm;
  unsigned long long* amax = reinterpret_cast<unsigned long long*>(p);
  LookAhead* la = nullptr;
  int rc = look_ahead(&la);
  if (!rc) rc = pivot_inverse_prepare();
  int sms = 0;
  if (!rc) rc = device_sm_count(&sms);
  if (rc) return rc;
  NED_CUDA(cudaMemsetAsync(amax, 0, sizeof(unsigned long long), st));
  const size_t nn = (size_t)n * n;
  amax_kernel<<<(int)((nn + 255) / 256 < 152 * 4 ? (nn + 255) / 256 : 152 * 4), 256, 0, st>>>(a, nn, amax);
  NED_LAUNCH_CHECK("amax_kernel");
  pad_identity_kernel<<<dim3(np, ceil_div(np, 1024)), 256, 0, st>>>(a, n, ap, np, amax, rowperm);
  NED_LAUNCH_CHECK("pad_identity_kernel");
  const int mtiles = np / 128, ntn = ceil_div(n, kTn);
  auto update = [&](int k0, int tiles, int jskip, int nskip, int ctas, cudaStream_t s) -> int {
    const int total = mtiles * tiles;
    if (total <= 0) return NEDMFT_OK;
    gj64_update_kernel<<<total < ctas ? total : ctas, 64 + 32 * kEpiW, USmem::kBytes, s>>>(
        ap, n, np, mtiles, tiles, total, k0, jskip, nskip, cimg, cexp, rimg, rexp, status);
    NED_LAUNCH_CHECK("gj64_update_kernel");
    return NEDMFT_OK;
  };
  auto panel = [&](int k0, cudaStream_t s) -> int {
    const int* in = nullptr;
    int count = n - k0, buf = 0;
    while (count > kPanRows) {  // rounds of 2048 rows until one cluster holds the candidates
      if (int e = launch_panel(ap, np, n, k0, in, count, cand[buf], false, pbuf, pimg, pexp, sw, rowperm, status, s))
        return e;
      in = cand[buf];
      count = ceil_div(count, kPanRows) * kNB;
      buf ^= 1;
    }
    return launch_panel(ap, np, n, k0, in, count, nullptr, true, pbuf, pimg, pexp, sw, rowperm, status, s);
  };
  constexpr int kFreeSms = 16;  // left to the window's and the panel's CTAs while the update runs
  if ((rc = panel(0, st))) return rc;
  for (int k0 = 0; k0 < n; k0 += kNB) {
    gj64_rpanel_kernel<<<dim3(2 * mtiles, 1), 512, RSmem::kBytes, st>>>(ap, np, mtiles, k0, pbuf, pimg, pexp, rimg,
                                                                        rexp, sw, cimg, cexp, status);
    NED_LAUNCH_CHECK("gj64_rpanel_kernel");
    const int k1 = k0 + kNB;
    if (k1 >= n) {
      if ((rc = update(k0, ntn, ntn, 0, sms, st))) return rc;
      break;
    }
    const int w0 = k1 / kTn, wn = ntn - w0 < 2 ? ntn - w0 : 2;  // the next panel's column tiles
    NED_CUDA(cudaEventRecord(la->panel, st));
    NED_CUDA(cudaStreamWaitEvent(la->side, la->panel, 0));
    if ((rc = update(k0, wn, 0, w0, sms, la->side))) return rc;
    if ((rc = panel(k1, la->side))) return rc;
    NED_CUDA(cudaEventRecord(la->chain, la->side));
    if ((rc = update(k0, ntn - wn, w0, wn, sms > 2 * kFreeSms ? sms - kFreeSms : sms, st))) return rc;
    NED_CUDA(cudaStreamWaitEvent(st, la->chain, 0));
  }
  unpermute_kernel<<<dim3(n, ceil_div(n, 1024)), 256, 0, st>>>(ap, np, n, rowperm, a, amax);
  NED_LAUNCH_CHECK("unpermute_kernel");
  return NEDMFT_OK;
}

}  // namespace nedmft
