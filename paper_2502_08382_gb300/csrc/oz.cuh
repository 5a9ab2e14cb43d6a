// FP64 products on the bf16 tensor cores by exact slicing (the Ozaki scheme), shared by the FP64 kernels that
// use it.
//
// A vector x (a row of the left operand or a column of the right one) is scaled by a power of two, |x_k| < 2^e,
// and every entry is rounded to 62 fractional bits, x_k = 2^(e - 62) I_k, and cut into eight balanced base-256
// digits, I_k = sum_p s_p 256^(7 - p), -128 <= s_p <= 127 (the leading one in [-64, 64]).  Each digit is exact in
// bf16.  The products of digits p of x and q of y with p + q = d <= 7 are summed over at most 128 entries in one
// FP32 accumulator: every partial sum is an integer of at most (d + 1) 128 2^14 <= 2^24, so the tensor cores' FP32
// accumulation is exact.  With hi = sum_{d <= 3} acc_d 2^(8 (3 - d)) and lo = sum_{d >= 4} acc_d 2^(8 (7 - d)) in
// 64-bit integers,
//   sum_k x_k y_k = 2^(e_x + e_y - 68) (2^32 hi + lo).
// Rounding to 62 bits costs 2^-63 of the largest entry in either factor, the dropped pairs (seven with p + q = 8, of at
// most 2^14 2^48 2^-124 each, and fewer beyond) at most 7.1 2^-62: a product of K entries lies within K 2^-58 2^(e_x + e_y)
// of the exact sum, against K 2^-53 for FP64 where all terms are of that size.
//
// A vector's entries share one exponent, so an entry far below the largest one keeps fewer than 53 bits.  Where the
// scales of a product's inner index are opposite on its two sides (a factor's inverse and a right-hand side: the one
// grows with the unknown's stiffness, the other falls), that would lose bits that FP64 keeps.  There both sides are
// cut with a shift s_k per inner index, x_k 2^-s_k and y_k 2^s_k (dig_key), which balances them; the shifts follow the
// unknowns' scales, so that the result is as independent of a power-of-two scaling of the unknowns as FP64's.
//
// All right-hand digits of one column block are stacked as the N rows of one operand (digit 0 first), so the MMA
// of left digit p with the stacked digits 0 .. 7 - p adds into the accumulators p .. 7, which lie side by side in
// TMEM: eight MMAs of N = 8 - p column blocks do all 36 products.
#pragma once
#include <cstdint>

#include "tc_common.cuh"

namespace feti {
namespace {

constexpr int kDig = 8;          // digits per FP64 value
constexpr int kDigK = 128;       // entries per exact accumulation
constexpr int kExpBad = 0x4000;  // "exponent" of a vector that holds an infinity or NaN
constexpr int kExpMin = -900;    // smallest exponent used (smaller vectors lose digits that underflow anyway)

// exponent e with |x| < 2^e from the largest high word (sign cleared) of a vector's entries
__device__ __forceinline__ int dig_exponent(uint32_t hi_max) {
  const int be = (int)(hi_max >> 20);
  return be == 0x7FF ? kExpBad : max(be - 1022, kExpMin);
}

// key of x 2^-s: its biased exponent minus s; the largest key of a vector gives its exponent
constexpr int kKeyZero = -(1 << 20), kKeyBad = 1 << 20;
__device__ __forceinline__ int dig_key(double x, int s) {
  const int be = (__double2hiint(x) >> 20) & 0x7FF;
  return be == 0 ? kKeyZero : be == 0x7FF ? kKeyBad : be - s;
}
__device__ __forceinline__ int dig_key_exponent(int key) {
  return key >= kKeyBad ? kExpBad : max(key - 1022, kExpMin);
}
// shift of a pivot x: its exponent if it is positive and normal, 0 otherwise; and half of it (for x a square)
__device__ __forceinline__ int dig_pivot_shift(double x) {
  const int be = __double2hiint(x) >> 20;
  return be <= 0 || be >= 0x7FF ? 0 : be - 1023;
}
__device__ __forceinline__ int dig_half_exponent(double x) {
  return dig_pivot_shift(x) >> 1;
}

// the digits of x (|x| < 2^e; |x| 2^-s < 2^e: cut with e + s) as signed bytes, digit 0 in the top byte
__device__ __forceinline__ uint64_t dig_cut(double x, int e) {
  const long long b = __double_as_longlong(x);
  const int be = (int)((b >> 52) & 0x7FF);
  if (be == 0 || be == 0x7FF) return 0;  // zero and subnormal; infinities and NaN are marked by the exponent
  const unsigned long long m = (unsigned long long)(b & 0xFFFFFFFFFFFFFLL) | (1ULL << 52);
  const int sh = be - 1023 - 52 + 62 - e;  // x = m 2^(be - 1075); |x| < 2^e gives sh <= 9
  long long I;
  if (sh >= 0) I = (long long)(m << sh);
  else if (sh > -54) I = (long long)((m + (1ULL << (-sh - 1))) >> -sh);
  else I = 0;
  if (b < 0) I = -I;
  return ((unsigned long long)I + 0x0080808080808080ULL) ^ 0x0080808080808080ULL;
}

// digit p of two packed values as a bf16 pair (low half: a)
__device__ __forceinline__ uint32_t dig_pair(uint64_t a, uint64_t b, int p) {
  const float fa = (float)(int)(signed char)(a >> (56 - 8 * p)), fb = (float)(int)(signed char)(b >> (56 - 8 * p));
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(fb), "f"(fa));
  return r;
}

// hi += / lo += of one element's eight accumulators (exact integers held as FP32)
__device__ __forceinline__ void dig_sum(const uint32_t (&a)[kDig], long long& hi, long long& lo) {
  int v[kDig];
#pragma unroll
  for (int d = 0; d < kDig; ++d) v[d] = __float2int_rn(__uint_as_float(a[d]));
  // v0 256 + v1 and v2 256 + v3 fit 32 bits (|v_d| <= (d + 1) 2^21)
  hi += (long long)(v[0] * 256 + v[1]) * 65536 + (v[2] * 256 + v[3]);
  lo += (long long)v[4] * (1 << 24) + (long long)v[5] * 65536 + (long long)v[6] * 256 + v[7];
}

// the value 2^ex (2^32 hi + lo) rounded to nearest, by integer arithmetic
__device__ __forceinline__ double dig_value(long long hi, long long lo, int ex) {
  hi += lo >> 32;
  uint32_t l = (uint32_t)lo;
  const bool neg = hi < 0;
  if (neg) {
    hi = ~hi + (l == 0);
    l = -l;
  }
  unsigned long long h = (unsigned long long)hi;
  if (h == 0) {
    h = l;
    l = 0;
    ex -= 32;
  }
  const int lz = __clzll((long long)h);
  const unsigned long long x = (unsigned long long)l << 32;
  const unsigned long long m = lz < 64 ? (h << lz) | (lz ? x >> (64 - lz) : 0ULL) : 0ULL;
  const unsigned long long mant = (m >> 11) + ((m >> 10) & 1);  // 53 bits, 2^52 <= mant <= 2^53
  const int e = 95 - lz + ex;                                   // value = mant 2^(e - 52)
  unsigned long long b = ((unsigned long long)(e + 1022) << 52) + mant;
  if (h == 0 || e < -1022) b = 0;  // subnormal results are flushed
  if (h != 0 && e > 1023) b = 0x7FF0000000000000ULL;  // (e = 1023 rounds up to infinity by itself)
  return __longlong_as_double((long long)(b | (neg ? 0x8000000000000000ULL : 0ULL)));
}

// 2^k for a normal exponent
__device__ __forceinline__ double dig_pow2(int k) { return __longlong_as_double((long long)(k + 1023) << 52); }

// bounded wait that also ends when another role has given up
__device__ __forceinline__ bool dig_wait(uint32_t mbar, uint32_t parity, volatile int* abort_flag) {
  for (int i = 0; i < (1 << 24); ++i) {
    if (mbar_test(mbar, parity)) return true;
    if ((i & 63) == 63) {
      if (*abort_flag) return false;
      __nanosleep(64);
    }
  }
  *abort_flag = 1;
  return false;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t& a, uint32_t& b, uint32_t& c, uint32_t& d) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
               : "r"(taddr));
}

}  // namespace
}  // namespace feti
