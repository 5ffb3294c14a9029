// Products of FP64 operands on the tensor cores.
//
// This part has two FP64 operations per clock per SM; an N x N product over m rows on them takes
// m N^2 / 2 clocks of one SM. Here an operand is a fixed-point number of 56 bits below a power of two
// above the largest entry of its row or column, cut into seven signed 8-bit digits, each an FP16
// integer of at most 128. Products of digits sum without rounding in the FP32 accumulators of tensor
// memory: with K <= 128 terms and at most seven digit pairs per level i + j = g, a level's sum is at most
// 7 x 128 x 2^14 < 2^24 whatever the operands. The levels 0 to 7 (34 digit products) are kept: what is left out
// is below 5 x 2^-64 of a full-scale term, an entry is cut at 2^-56 of its row's or column's largest and a sum
// at 2^-56 of a full-scale term, so that a product is as good as one in FP64 in norm: an FP64 sum's terms and
// partial sums are rounded at 2^-53 of themselves. Entry by entry it is not: entries below an eighth of their
// row's or column's largest hold fewer than 53 bits, and a sum of such entries only (a member much smaller
// than the others, in the products whose scales run across members) loses those bits. (With the levels 0 to 6
// and sums cut downwards at 2^-53 the analysis at m = 10,000, N = 100 lost a digit: 3.8e-14 against 2.3e-15;
// with these it is 1.9e-15 off.) A sum leaves tensor memory as integers, and becomes an FP64
// number with integer operations only: conversions and scalings on the FP64 unit would take longer
// than the products.
//
// Infinities and NaN: the scale of their row or column is not finite, and its results are NaN.
#pragma once

#include "krylov.cuh"

namespace enkf {

constexpr int kDg = 7;        // digits
constexpr int kDl = 8;        // levels
constexpr int kDR = 80;       // rows per tile: ten groups of eight
constexpr int kDT = 640;      // threads: one item (eight columns of a row) each per 64 columns of a tile

// High word of |x|: orders like |x|, and its exponent field is the scale's.
__device__ __forceinline__ int dg_abs_hi(double x) { return __double2hiint(x) & 0x7FFFFFFF; }
// Exponent field E of a scale: entries are below 2^(E - 1022). 2047: an infinity or NaN is among them.
__device__ __forceinline__ int dg_exp(int abs_hi) { return max(abs_hi >> 20, 64); }

// x 2^-(E - 1022) in units of 2^-55, rounded
__device__ __forceinline__ int64_t dg_fixed(double x, int E) {
  const int64_t b = __double_as_longlong(x);
  const int ex = (int)(b >> 52) & 2047, d = min(max(E - ex, 0), 62);
  const int64_t y = ((b & 0xFFFFFFFFFFFFFll) | (1ll << 52)) << 2;   // (a subnormal is cut to zero: E >= 64)
  const int64_t v = (y + ((1ll << d) >> 1)) >> d;
  return b < 0 ? -v : v;
}
// The digits of eight numbers along the 16-byte direction of a core row, weights 2^-7, 2^-15, ... 2^-55,
// as FP16: 1024 + n has the bits 0x6400 + n, so a byte biased by 128 becomes a digit with one subtraction.
struct Digits8 {
  uint4 w[kDg];
  __device__ __forceinline__ void make(const double (&x)[8], const int (&E)[8]) {
    uint32_t u[kDg][4];
    const __half2 bias = __halves2half2(__ushort_as_half((unsigned short)0x6480), __ushort_as_half((unsigned short)0x6480));
    auto put = [&](int g, int q, uint32_t v) {
      const __half2 h = __hsub2(*reinterpret_cast<const __half2*>(&v), bias);
      u[g][q] = *reinterpret_cast<const uint32_t*>(&h);
    };
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      // every digit biased by 128
      const int64_t a = dg_fixed(x[2 * q], E[2 * q]) + 0x0080808080808080ll, b = dg_fixed(x[2 * q + 1], E[2 * q + 1]) + 0x0080808080808080ll;
      const uint32_t al = (uint32_t)a, bl = (uint32_t)b, ah = (uint32_t)(a >> 32), bh = (uint32_t)(b >> 32);
      put(0, q, __byte_perm(ah, bh, 0x7632) | 0x64006400u);   // bits 48 on: 0 .. 256
      put(1, q, (__byte_perm(ah, bh, 0x0501) & 0x00FF00FFu) | 0x64006400u);
      put(2, q, (__byte_perm(ah, bh, 0x0400) & 0x00FF00FFu) | 0x64006400u);
      put(3, q, (__byte_perm(al, bl, 0x0703) & 0x00FF00FFu) | 0x64006400u);
      put(4, q, (__byte_perm(al, bl, 0x0602) & 0x00FF00FFu) | 0x64006400u);
      put(5, q, (__byte_perm(al, bl, 0x0501) & 0x00FF00FFu) | 0x64006400u);
      put(6, q, (__byte_perm(al, bl, 0x0400) & 0x00FF00FFu) | 0x64006400u);
    }
#pragma unroll
    for (int g = 0; g < kDg; ++g) w[g] = make_uint4(u[g][0], u[g][1], u[g][2], u[g][3]);
  }
  __device__ __forceinline__ void store(unsigned char* at, int digit_bytes) const {
#pragma unroll
    for (int g = 0; g < kDg; ++g) *reinterpret_cast<uint4*>(at + g * digit_bytes) = w[g];
  }
};

// The value of an entry from its levels: in units of 2^-55 of the product of the scales
template <int LC>
__device__ __forceinline__ int64_t dg_join(const float (&a)[kDl][LC], int q) {
  auto n = [&](int g) { return (int64_t)__float2int_rn(a[g][q]); };
  const int64_t hi = (n(0) << 24) + (n(1) << 16) + (n(2) << 8) + n(3);   // at most 2^45.1 (K <= 128)
  const int64_t lo = (n(4) << 24) + (n(5) << 16) + (n(6) << 8) + n(7);
  return (hi << 17) + ((lo + (1 << 14)) >> 15);
}
// ... and as FP64, rounded to nearest (ties away), with the scales' exponent fields
__device__ __forceinline__ double dg_value(int64_t x, int ea, int eb) {
  const uint64_t v = x < 0 ? (uint64_t)-x : (uint64_t)x;
  const int lz = __clzll((long long)v);
  const uint64_t n = v << (lz & 63), man = (n >> 11) + ((n >> 10) & 1u);
  const int e = 1023 + 63 - 55 - 2 * 1022 + ea + eb - lz;   // exponent field
  uint64_t bits = ((uint64_t)(e - 1) << 52) + man;
  if (v == 0 || e <= 0) bits = 0;
  if (e >= 2047) bits = 0x7FF0000000000000ull;
  if (max(ea, eb) == 2047) bits = 0x7FF8000000000000ull;
  return __longlong_as_double((long long)(bits | ((uint64_t)x & 0x8000000000000000ull)));
}

// The digit products of D = A B (M = 128, 64 columns), level g = i + j <= 7 in the columns at d + 64 g, over ks
// blocks of 16 along K. The digits of B lie one behind the other along N (B_SL bytes), so that up to four of
// them share an MMA (135 cycles for 256 columns, 64 for 64). Called by one whole warp, `lead` on one lane.
template <bool AMN, bool BMN, int A_PART, int A_STEP, int B_SL, int B_STEP>
__device__ __forceinline__ void dg_issue(uint32_t d, uint64_t a, uint64_t b, int ks, bool acc, uint64_t* mbar, uint32_t lead) {
  asm volatile("" : "+l"(a), "+l"(b), "+r"(d));   // recomputed per tile instead of held in registers
#pragma unroll 1
  for (int kb = 0; kb < ks; ++kb) {
#pragma unroll
    for (int i = 0; i < kDg; ++i) {
      auto mma = [&](int j0, int nj) {
        // (i, j0) starts its level's sum when i = 0, and (1, 6) the last level's
        const bool add = acc || kb > 0 || (i > 0 && !(i == 1 && j0 == 6));
        umma_lead(d + (uint32_t)((i + j0) * 64), a + (uint64_t)((i * A_PART) >> 4), b + (uint64_t)((j0 * B_SL) >> 4),
                  sl_idesc(nj * 64, AMN, BMN), add ? 1u : 0u, lead);
      };
      const int n = kDl - i < kDg ? kDl - i : kDg;   // digits of B: 7, 7, 6, 5, ...
      if (i == 1) {
        mma(0, 3);
        mma(3, 3);
        mma(6, 1);
      } else {
        const int first = n > 4 ? (n + 1) / 2 : n;
        mma(0, first);
        if (first < n) mma(first, n - first);
      }
    }
    a += (uint64_t)(A_STEP >> 4);
    b += (uint64_t)(B_STEP >> 4);
  }
  if (lead) umma_commit(mbar);
}

}  // namespace enkf
