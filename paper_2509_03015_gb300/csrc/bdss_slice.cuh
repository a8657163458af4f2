// Products of FP64 and FP32 tiles on the tcgen05 tensor cores at their full
// accuracy, with the operands cut into parts inside the kernel that uses them
// (nothing of the parts goes to memory).
//
// FP64.  A row of K <= 64 operand entries gets one binary exponent, the
// largest of its entries, and every entry becomes the signed integer
//   q = trunc(v 2^-(exponent) 2^62),
// written in kDig = 8 base-256 digits q = sum_p d_p 256^(7-p) with
// -128 <= d_p <= 127 and |d_0| <= 64, each exact in FP16.  The product of two
// rows is then
//   sum_k q_a q_b = sum_t 256^(14 - t) ACC_t,
//   ACC_t = sum_{p+q=t} sum_k d_p(a) d_q(b),
// and only the diagonals t < 8 are formed: the digit pairs left out weigh
// below 2^-64 x 64 x 8, i.e. 2^-57 of the product of the two row maxima at
// worst and 2^-61 for digits of random sign.  Every
// |ACC_t| <= 2 x 64 x 64 x 128 + (t - 1) x 64 x 128 x 128 < 2^23, so the FP32
// accumulation of the tensor cores is exact whatever its order.
//
// FP32.  An entry is the sum of kDig = 3 BF16 numbers: h, its rounding to a
// multiple of 2^-8 times the power of two above the row's largest entry, and
// two roundings of what is left (25 bits or more below the row maximum).  The
// products of parts p + q <= 2 are summed, each p + q in an accumulator of its
// own; the ones left out are below 2^-26 of the product of the row maxima.  The
// tensor cores truncate where they add in FP32, which on sums of 256 BF16
// products cost three bits against a chain of FP32 multiply-adds; the sum of
// the products h h is an integer below 2^16 x 64 and exact, and the others'
// truncation weighs 2^-8 as much.
//
// Scaling along K.  These bounds are relative to the row maxima, so they say
// nothing about a product whose rows have their large entries at different K
// indices.  State components in different units do that: with the states of a
// block scaled by s_k a coupling's entry k grows with s_k and that of the
// inverse factor with 1 / s_k (spread 1e8: 5e-11 of the solution lost).  So
// before it is cut, entry k of one operand is scaled by 2^-e_k and of the other
// by 2^e_k, exactly, with 2^e_k about the square root of the diagonal entry
// that index k belongs to (sl_half_exp).  The rows of an SPD system's
// off-diagonal blocks are then bounded by the other index's diagonal entry
// alone, |a_rk| <= sqrt(a_rr a_kk), whatever the units, as the error of a
// Cholesky factorisation is.  Products of W^T and of y with each other need no
// scaling: their K indices are rows of L^{-1} A and carry no unit.
//
// One tcgen05.mma (kind::f16, M = 128) per A part p and K step of 16 covers
// the B parts q = 0 .. kDig-1-p of up to 32 B rows at once: the B operand
// stacks the parts (32 rows each), and its D columns start at 32 p, so the
// pair (p, q) lands on the columns of diagonal p + q.  p = 0 covers every
// diagonal, so its first K step clears the accumulators.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "bdss_tc.cuh"

namespace bdss {

template <typename T> struct SliceFmt;
template <> struct SliceFmt<double> { static constexpr int kDig = 8; };
template <> struct SliceFmt<float> { static constexpr int kDig = 3; };

constexpr int kSlRows = 128;             // A rows of a tile (TMEM lanes)
constexpr int kSlK = 64;                 // K entries of a tile (128 bytes of FP16)
constexpr int kSlCols = 32;              // B rows of a column tile
constexpr int kSlASlab = kSlRows * 128;  // bytes of one digit of the A tile
constexpr int kSlBSlab = kSlCols * 128;  // bytes of one digit of a B tile

// Exponent field of |v| (0 for zero and subnormals: they count as zero).
__device__ __forceinline__ int sl_exp(double v) { return (__double2hiint(v) >> 20) & 0x7FF; }
__device__ __forceinline__ int sl_exp(float v) { return (__float_as_int(v) >> 23) & 0xFF; }
// The row exponent that enters sl_value: a row with an infinity or NaN poisons
// every product it takes part in, as a floating-point product would.
constexpr int kSlPoisonEx = 1 << 16;
template <typename T>
__device__ __forceinline__ int sl_row_exp(int ex) {
  return sizeof(T) == 8 && ex == 0x7FF ? kSlPoisonEx : ex;
}
// e with 2^e <= sqrt(x) < 2^(e+1) for a positive normal x (any bits: -512 <= e <= 512).
__device__ __forceinline__ int sl_half_exp(double x) { return (sl_exp(x) - 1023) >> 1; }
__device__ __forceinline__ int sl_half_exp(float x) { return (sl_exp(x) - 127) >> 1; }
// v 2^e, exactly; FP64: on the integer pipe, a subnormal operand or result is
// zero, as in the cut.
__device__ __forceinline__ double sl_scale(double v, int e) {
  const int ex = sl_exp(v), x = ex + e;
  if ((unsigned)(ex - 1) < 0x7FEu && (unsigned)(x - 1) < 0x7FEu)
    return __hiloint2double(__double2hiint(v) + (int)((unsigned)e << 20), __double2loint(v));
  if (ex == 0x7FF) return v;
  return ex == 0 || x <= 0 ? 0.0 : copysign(__longlong_as_double(0x7FF0000000000000LL), v);
}
__device__ __forceinline__ float sl_scale(float v, int e) { return v * __int_as_float((127 + e) << 23); }
// Entries that count as v 2^e.  FP32 scales them first (sl_prep).  FP64 leaves
// the bits alone (an FP64 instruction holds a warp's FP64 unit for 64 cycles on
// this GPU): their exponent fields and shifts are offset instead.
__device__ __forceinline__ void sl_prep(double &, int) {}
__device__ __forceinline__ void sl_prep(float &v, int e) { v = sl_scale(v, e); }
// Exponent of such an entry, poison included; a row's largest is its row
// exponent as it is.  A zero counts as 2^(e - 1023) <= 2^-511 in it, which is
// nothing beside the sqrt(a_rr) that a row of an SPD system's factorisation is
// rounded against; where rows have no such bound, sl_exp_nz leaves zeros out.
__device__ __forceinline__ int sl_exp_at(double v, int e) {
  const int x = sl_exp(v);
  return x + (x == 0x7FF ? kSlPoisonEx : e);
}
__device__ __forceinline__ int sl_exp_at(float v, int) { return sl_exp(v); }
constexpr int kSlNoEx = -(1 << 13);  // below every exponent
__device__ __forceinline__ int sl_exp_nz(double v, int e) { return sl_exp(v) == 0 ? kSlNoEx : sl_exp_at(v, e); }

// Biased digits of v under the row exponent field exmax: the byte p from the
// top is d_p + 128.
__device__ __forceinline__ unsigned long long sl_biased(double v, int exmax) {
  const long long b = __double_as_longlong(v);
  const int ex = (int)(b >> 52) & 0x7FF;
  unsigned long long m = ((unsigned long long)(b & 0xFFFFFFFFFFFFFLL) | 0x10000000000000ULL) << 9;
  const int s = exmax - ex;
  m = (ex == 0) ? 0ULL : (m >> (s > 63 ? 63 : s));
  return (b < 0 ? 0ULL - m : m) + 0x8080808080808080ULL;
}
// Two digits (bytes lo and hi of each half of c) as FP16 pairs: 0x6400 | b is
// 1024 + b, and subtracting 1152 leaves d = b - 128, both exact.
__device__ __forceinline__ void sl_half_pairs(unsigned c, unsigned &lo, unsigned &hi) {
  const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));
  unsigned l = __byte_perm(c, 0x64646464u, 0x4240), h = __byte_perm(c, 0x64646464u, 0x4341);
  __half2 a = *reinterpret_cast<__half2 *>(&l), b = *reinterpret_cast<__half2 *>(&h);
  a = __hsub2(a, bias);
  b = __hsub2(b, bias);
  lo = *reinterpret_cast<unsigned *>(&a);
  hi = *reinterpret_cast<unsigned *>(&b);
}

// Two consecutive K entries of one row -> 4 bytes of every digit slab.
// e0, e1: they count as v0 2^e0, v1 2^e1 (FP32: scaled already).
template <typename T>
__device__ __forceinline__ void sl_store2(T v0, T v1, int exmax, unsigned char *dst, int stride, int e0 = 0, int e1 = 0);
template <>
__device__ __forceinline__ void sl_store2<double>(double v0, double v1, int exmax, unsigned char *dst, int stride,
                                                  int e0, int e1) {
  const unsigned long long u0 = sl_biased(v0, exmax - e0), u1 = sl_biased(v1, exmax - e1);
  const unsigned h0 = (unsigned)(u0 >> 32), h1 = (unsigned)(u1 >> 32), l0 = (unsigned)u0, l1 = (unsigned)u1;
  unsigned w[8];
  sl_half_pairs(__byte_perm(h0, h1, 0x7632), w[1], w[0]);
  sl_half_pairs(__byte_perm(h0, h1, 0x5410), w[3], w[2]);
  sl_half_pairs(__byte_perm(l0, l1, 0x7632), w[5], w[4]);
  sl_half_pairs(__byte_perm(l0, l1, 0x5410), w[7], w[6]);
#pragma unroll
  for (int p = 0; p < 8; ++p) *reinterpret_cast<unsigned *>(dst + p * stride) = w[p];
}
// The BF16 parts of two entries, one pair per part.
__device__ __forceinline__ void sl_parts(float v0, float v1, int exmax, unsigned (&w)[3]) {
  // adding 1.5 x 2^23 units rounds to the unit (2^-7 of the row exponent)
  const float C = __int_as_float((min(exmax + 16, 254) << 23) | 0x400000);
  float h0 = (v0 + C) - C, h1 = (v1 + C) - C;
#pragma unroll
  for (int p = 0; p < 3; ++p) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(h0, h1);
    w[p] = *reinterpret_cast<const unsigned *>(&h);
    v0 -= __low2float(h);
    v1 -= __high2float(h);
    h0 = v0;
    h1 = v1;
  }
}
template <>
__device__ __forceinline__ void sl_store2<float>(float v0, float v1, int exmax, unsigned char *dst, int stride, int,
                                                 int) {
  unsigned w[3];
  sl_parts(v0, v1, exmax, w);
#pragma unroll
  for (int p = 0; p < 3; ++p) *reinterpret_cast<unsigned *>(dst + p * stride) = w[p];
}

// Byte offset of 16-byte group g (K entries 8 g .. 8 g + 7) of row r in a
// 128-byte-swizzled slab.
__device__ __forceinline__ int sl_off(int r, int g) { return r * 128 + ((g ^ (r & 7)) << 4); }

// D = FP32, A = B = FP16 (FP64 digits) or BF16 (FP32 parts), both K-major, M = 128 x N.
template <typename T>
__host__ __device__ constexpr uint32_t sl_idesc(int N) {
  return (1u << 4) | (sizeof(T) == 4 ? (1u << 7) | (1u << 10) : 0u) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kSlRows >> 4) << 24);
}

__device__ __forceinline__ void sl_mma(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool sl_elect() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// All digit pairs of A (128 rows) times a B tile of `cols` rows (16 or 32), K
// steps 0 .. ks - 1, into the accumulators at TMEM address d (diagonal t at
// columns cols t ..).  One elected lane of a warp that takes this path as a
// whole (its operands then stay in uniform registers: issued by one thread of
// a diverged warp, a product took 130 cycles against the tensor core's 72);
// rolled over p, since the code of the digit kernels has to stay in the
// instruction cache.
template <typename T>
__device__ __forceinline__ void sl_issue(uint32_t d, const unsigned char *A, const unsigned char *B, int cols, int ks) {
  constexpr int kDig = SliceFmt<T>::kDig;
  const uint64_t ad0 = tc_desc_sw128(A, 0), bd0 = tc_desc_sw128(B, 0);
#pragma unroll 1
  for (int p = 0; p < kDig; ++p) {
    const uint32_t idesc = sl_idesc<T>(cols * (kDig - p)), dp = d + (uint32_t)(cols * p);
    // the start address field counts 16-byte units: a slab is kSlASlab / 16,
    // a K step of 16 FP16 entries 2 of them
    const uint64_t ad = ad0 + (uint64_t)(p * (kSlASlab / 16));
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < ks) sl_mma(dp, ad + 2 * k, bd0 + 2 * k, idesc, (uint32_t)(p | k));
  }
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t (&r)[4]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// An accumulator entry as an integer without the conversion unit (16 lanes a
// cycle and SM): |x| <= 2^22, adding 1.5 * 2^23 puts x in the binade of unit
// spacing, and the bits are kSlBias + x.  |x| < 2^23: 1.5 * 2^24 and a spacing of
// two (bits kSlBias2 + x / 2), which rounds the last bit away -- used for the
// two lowest diagonals, where it weighs 2^-60 of the product of the row maxima.
constexpr unsigned kSlBias = 0x4B400000u, kSlBias2 = 0x4BC00000u;
__device__ __forceinline__ unsigned sl_bits22(float x) { return (unsigned)__float_as_int(x + 12582912.0f); }
__device__ __forceinline__ unsigned sl_bits23(float x) { return (unsigned)__float_as_int(x + 25165824.0f); }

// (-1)^neg (m2 2^64 + m1 2^32 + m0) 2^S rounded to FP64, whatever the range
// (zero, subnormal and infinite results; a poisoned row's exponent is out of it).
static __device__ __noinline__ double sl_value_slow(unsigned m2, unsigned m1, unsigned m0, bool neg, int S) {
  if (S > kSlPoisonEx / 2) return __longlong_as_double(0x7FF8000000000000LL);
  if ((m2 | m1 | m0) == 0u) return 0.0;
  unsigned long long hi = ((unsigned long long)m2 << 32) | m1;
  double r;
  if (hi == 0) {
    r = scalbn((double)m0, S);
  } else {  // 64 leading bits, the last one sticky
    const int lz = __clzll((long long)hi);
    unsigned long long m = lz == 0 ? hi : (hi << lz) | (((unsigned long long)m0 << 32) >> (64 - lz));
    if (lz < 32 && (unsigned)(m0 << lz) != 0u) m |= 1ULL;
    r = scalbn(__ull2double_rn(m), S + 32 - lz);
  }
  return neg ? -r : r;
}

// sum_t ACC_t 256^(7-t) 2^(exa + exb - 2112), rounded once to FP64 on the
// integer pipes (an FP64 instruction holds a warp's FP64 unit for 64 cycles on
// this GPU).  With |d_0| <= 64 the diagonals are at most 2^18, 2^20, 2^21,
// 3 2^20, ..., 7 2^20, so neighbouring pairs combine in 32 bits.
//
// The logic pipe (half rate) sets the pace of the drains, so additions that
// can be multiply-adds are, the biases of the pairs are subtracted once, the
// sign is taken off by complement (one unit of 2^-62 of the row maxima), and
// everything unusual goes to sl_value_slow: about 30 logic instructions an
// entry, half of a conversion through 64-bit shifts and selects (the products
// of a 128 x 64 tile took 9,200 of a round's 24,700 cycles to drain).
__device__ __forceinline__ double sl_value(const float (&c)[8], int exa, int exb) {
  const int h01 = (int)(sl_bits22(c[0]) * 256u + sl_bits22(c[1]) - kSlBias * 257u);
  const int h23 = (int)(sl_bits22(c[2]) * 256u + sl_bits22(c[3]) - kSlBias * 257u);
  const int h45 = (int)(sl_bits22(c[4]) * 256u + (unsigned)__float2int_rn(c[5]) - kSlBias * 256u);
  const int h67 = (int)(sl_bits23(c[6]) * 512u + sl_bits23(c[7]) * 2u - kSlBias2 * 514u);
  const long long H = (long long)h01 * 65536 + h23, L = (long long)h45 * 65536 + h67;
  const long long hi = H + (int)(L >> 32);  // value = (hi 2^32 + lo) 2^S
  const int sgn = (int)(hi >> 63);
  const unsigned m2 = (unsigned)((int)(hi >> 32) ^ sgn), m1 = (unsigned)((int)hi ^ sgn), m0 = (unsigned)((int)L ^ sgn);
  // 96 bits; the leading word is m2 or m1
  const bool p = m2 != 0;
  const unsigned w2 = p ? m2 : m1, w1 = p ? m1 : m0, w0 = p ? m0 : 0u;
  const int z = __clz((int)w2);
  const unsigned a1 = __funnelshift_l(w1, w2, z), a0 = __funnelshift_l(w0, w1, z);
  // exponent field of the result, less one: the mantissa's leading bit adds it
  const int S = exa + exb - 2112, be = S + (p ? 1023 + 95 - 1 : 1023 + 63 - 1) - z;
  if (w2 == 0u || (unsigned)be > 2044u) return sl_value_slow(m2, m1, m0, sgn != 0, S);
  const unsigned t0 = __funnelshift_r(a0, a1, 11), rb = (a0 >> 10) & 1u;
  const unsigned long long bits =
      (((unsigned long long)((unsigned)be * 0x100000u + (a1 >> 11)) << 32) | t0) + rb;  // a carry raises the exponent
  return __longlong_as_double((long long)(bits | ((unsigned long long)((unsigned)sgn & 0x80000000u) << 32)));
}
// The same for FP32: the smaller parts' products first.
__device__ __forceinline__ float sl_value(const float (&c)[3], int, int) { return c[0] + (c[1] + c[2]); }

}  // namespace bdss
