#pragma once
// FP64 products on the tensor cores, by exact fixed-point digits.
//
// GB300 runs one FP64 FMA warp instruction per 16 cycles and SM (2 FMAs per
// cycle; its FP64 tensor form m8n8k4 runs at the same rate) but 1024
// half-precision FMAs per cycle through mma.sync m16n8k16.  So a product of
// FP64 matrices is formed from integers (the error-free splitting of Ozaki,
// Ogita, Oishi & Rump, Numer. Algorithms 59 (2012)): every element is rounded
// once to X 2^{E-62}, X a 63-bit integer, E an exponent its row, column or
// matrix shares, and X = sum_i d_i 256^{7-i} with eight digits d_i in
// -128..127.  Digits are exact in FP16, a product of two is an integer below
// 2^14, and the MMA's FP32 accumulators stay below 2^24 while at most 128
// products of at most eight digit pairs add up: every sum is exact.  The
// digit pairs with i + j <= 7 are formed (36 MMAs per 16-deep step); the rest
// lies below 2^-58 of the operands' scale.  The integer sums are put together
// in 96 bits and rounded once to FP64.  So the error is an absolute one of
// about 2^-60 of (row scale) x (column scale) per term plus half an ulp of the
// result, where an FMA chain of K terms loses about sqrt(K) half ulps of its
// partial sums.  An element below 2^-9 of its scale keeps fewer than 53 bits,
// and subnormal FP64 values count as zero: an operand whose rows or columns
// differ in size and must keep their own precision takes an exponent for each.
//
// Rate: 36 MMAs of 2048 FMAs replace 2048 FP64 FMAs: 72 cycles per SM (measured:
// 2.00 per MMA; the INT8 form m16n8k32 takes 16.3) against 1024.  Around it, digits are made once per element (about 15 integer
// operations), taken apart into half2 fragments (2.5 operations per digit
// pair) and put together (about 40 operations per output).
//
// A packed element is X + 0x8080808080808080: byte 7 - i is d_i + 128.
// NaN and infinities: an operand that holds one gets the exponent kDigitBad,
// and every product with it is NaN.
#include <cuda_fp16.h>
#include <stdint.h>

#include "chain.h"

namespace pqmc {

// smallest E with |x| < 2^E
static __device__ __forceinline__ int digit_exp(double x) {
  const int e = (__double2hiint(x) >> 20) & 0x7ff;
  return e == 0x7ff ? kDigitBad : e == 0 ? kDigitNone : e - 1022;
}
static __device__ __forceinline__ int digit_exp(float x) {
  const int e = (__float_as_int(x) >> 23) & 0xff;
  return e == 0xff ? kDigitBad : e == 0 ? (x != 0.f ? -125 : kDigitNone) : e - 126;
}

// packed digits of x = m 2^{q} (m the integer significand) against exponent E
static __device__ __forceinline__ unsigned long long digit_pack(unsigned long long m, int q, int E, bool neg) {
  const int sh = q + 62 - E;                             // X = m 2^sh
  unsigned long long X;
  if (sh >= 0) X = m << (sh & 63);                       // |x| < 2^E: at most 2^62
  else if (sh < -60) X = 0;
  else X = ((m >> (-sh - 1)) + 1) >> 1;                  // to nearest
  return (neg ? 0ull - X : X) + kDigitZero;
}
static __device__ __forceinline__ unsigned long long digit_pack(double x, int E) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  if (e == 0 || e == 0x7ff) return kDigitZero;           // (subnormals count as zero)
  return digit_pack((b & 0xfffffffffffffull) | 0x10000000000000ull, e - 1075, E, (long long)b < 0);
}
static __device__ __forceinline__ unsigned long long digit_pack(float x, int E) {
  const unsigned b = (unsigned)__float_as_int(x);
  const int e = (int)(b >> 23) & 0xff;
  if (e == 0xff) return kDigitZero;
  const unsigned m = e ? ((b & 0x7fffffu) | 0x800000u) : (b & 0x7fffffu);
  return digit_pack((unsigned long long)m, (e ? e : 1) - 150, E, (int)b < 0);
}

// (hi 2^32 + lo) 2^e rounded to FP64 (|hi| < 2^60)
static __device__ __forceinline__ double digit_value(long long hi, long long lo, int e) {
  hi += lo >> 32;
  unsigned l = (unsigned)lo;
  const bool neg = hi < 0;
  if (neg) {
    hi = ~hi;
    l = ~l;
    if (++l == 0) ++hi;
  }
  if (hi == 0) {
    if (l == 0) return 0.0;
    hi = (long long)l;
    l = 0;
    e -= 32;
  }
  const int z = __clzll(hi);
  unsigned long long m = (unsigned long long)hi << z;
  m |= z >= 32 ? (unsigned long long)l << (z - 32) : (unsigned long long)(l >> (32 - z));
  // value = m 2^{e + 32 - z}, bit 63 of m set; 53 bits stay
  m += 0x400ull;
  int E = e + 32 - z + 63;
  if ((long long)m >= 0) {                               // rounded up to the next power of two
    m = 0x8000000000000000ull;
    ++E;
  }
  if (E < -1022) return 0.0;
  if (E > 1023) return __longlong_as_double(neg ? 0xfff0000000000000ll : 0x7ff0000000000000ll);
  const unsigned long long b = ((unsigned long long)(E + 1022) << 52) + (m >> 11);
  return __longlong_as_double((long long)(neg ? b | 0x8000000000000000ull : b));
}

// digit pairs of two packed elements (k, k + 1) as half2 d_i, i = 0..7
static __device__ __forceinline__ void digit_halves(unsigned long long y0, unsigned long long y1, uint32_t h[8]) {
  const uint32_t a[2] = {(uint32_t)(y0 >> 32), (uint32_t)y0}, b[2] = {(uint32_t)(y1 >> 32), (uint32_t)y1};
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0xe480));   // -1152: (1024 + byte) - 1152
#pragma unroll
  for (int w = 0; w < 2; ++w) {
    const uint32_t p = __byte_perm(a[w], b[w], 0x6273), q = __byte_perm(a[w], b[w], 0x4051);
    const uint32_t v[4] = {__byte_perm(p, 0x64646464u, 0x4140), __byte_perm(p, 0x64646464u, 0x4342),
                           __byte_perm(q, 0x64646464u, 0x4140), __byte_perm(q, 0x64646464u, 0x4342)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      __half2 t;
      *reinterpret_cast<uint32_t*>(&t) = v[i];
      t = __hadd2(t, off);
      h[4 * w + i] = *reinterpret_cast<uint32_t*>(&t);
    }
  }
}

static __device__ __forceinline__ void digit_mma(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                 uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// C = A B by one CTA (every thread calls; no barrier inside): A(i, k) =
// A[i sai + k sak], B(k, j) = B[j sbj + k sbk] packed digits; kAk (kBk): k
// contiguous in A (B), sak = 1 (sbk = 1) and rows 16-byte aligned.  ea(i), eb(j):
// exponents.  epi(i, j, value) for every element; with upper, only the 16 x 8
// tiles that reach j >= i; with btri, B(k, j) = 0 for k > j is left out.  One
// warp per tile, its 36 digit-pair sums in 32 accumulator registers.
template <bool kAk, bool kBk, typename EA, typename EB, typename Epi>
__device__ __forceinline__ void digit_gemm(int M, int Nn, int K, const unsigned long long* A, int sai, int sak,
                                           const unsigned long long* B, int sbj, int sbk, EA ea, EB eb, bool upper, bool btri, Epi epi) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int tm = (M + 15) >> 4, tn = (Nn + 7) >> 3;
  int m0 = 0, n0 = 8 * (int)(threadIdx.x >> 5);
  const int hop = 8 * (int)(blockDim.x >> 5);
  for (;; n0 += hop) {
    while (n0 >= 8 * tn) { n0 -= 8 * tn; m0 += 16; }
    if (m0 >= 16 * tm) break;
    if (upper && n0 + 7 < m0) continue;
    const int r0 = min(m0 + g, M - 1), r1 = min(m0 + g + 8, M - 1), cj = min(n0 + g, Nn - 1);
    const unsigned long long* pa0 = A + (long)r0 * sai;
    const unsigned long long* pa1 = A + (long)r1 * sai;
    const unsigned long long* pb = B + (long)cj * sbj;
    long long hi[4] = {0, 0, 0, 0}, lo[4] = {0, 0, 0, 0};
    const int kn = btri ? min(K, n0 + 8) : K;
    for (int kc = 0; kc < kn; kc += 128) {               // sums stay exact over 128 terms
      float acc[8][4];
#pragma unroll
      for (int d = 0; d < 8; ++d) acc[d][0] = acc[d][1] = acc[d][2] = acc[d][3] = 0.f;
      const int ke = min(kc + 128, kn);
#pragma unroll 1
      for (int k0 = kc; k0 < ke; k0 += 16) {
        const int k = k0 + 2 * t;
        unsigned long long ya[8], yb[4];
        if (k0 + 16 <= K) {
          if (kAk) {
            const ulonglong2 v0 = *reinterpret_cast<const ulonglong2*>(pa0 + k), v1 = *reinterpret_cast<const ulonglong2*>(pa1 + k);
            const ulonglong2 v2 = *reinterpret_cast<const ulonglong2*>(pa0 + k + 8), v3 = *reinterpret_cast<const ulonglong2*>(pa1 + k + 8);
            ya[0] = v0.x; ya[1] = v0.y; ya[2] = v1.x; ya[3] = v1.y; ya[4] = v2.x; ya[5] = v2.y; ya[6] = v3.x; ya[7] = v3.y;
          } else {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              ya[e] = pa0[(long)(k + e) * sak];
              ya[2 + e] = pa1[(long)(k + e) * sak];
              ya[4 + e] = pa0[(long)(k + 8 + e) * sak];
              ya[6 + e] = pa1[(long)(k + 8 + e) * sak];
            }
          }
          if (kBk) {
            const ulonglong2 w0 = *reinterpret_cast<const ulonglong2*>(pb + k), w1 = *reinterpret_cast<const ulonglong2*>(pb + k + 8);
            yb[0] = w0.x; yb[1] = w0.y; yb[2] = w1.x; yb[3] = w1.y;
          } else {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              yb[e] = pb[(long)(k + e) * sbk];
              yb[2 + e] = pb[(long)(k + 8 + e) * sbk];
            }
          }
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int kk = k + (e & 1) + 8 * (e >> 1);
            const bool in = kk < K;
            ya[4 * (e >> 1) + (e & 1)] = in ? pa0[(long)kk * sak] : kDigitZero;
            ya[4 * (e >> 1) + 2 + (e & 1)] = in ? pa1[(long)kk * sak] : kDigitZero;
            yb[e] = in ? pb[(long)kk * sbk] : kDigitZero;
          }
        }
        uint32_t b0[8], b1[8], a0[8], a1[8], a2[8], a3[8];
        digit_halves(yb[0], yb[1], b0);
        digit_halves(yb[2], yb[3], b1);
        digit_halves(ya[0], ya[1], a0);
        digit_halves(ya[2], ya[3], a1);
        digit_halves(ya[4], ya[5], a2);
        digit_halves(ya[6], ya[7], a3);
#pragma unroll
        for (int i = 0; i < 8; ++i)
#pragma unroll
          for (int j = 0; j < 8 - i; ++j) digit_mma(acc[i + j], a0[i], a1[i], a2[i], a3[i], b0[j], b1[j]);
      }
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        hi[r] += ((long long)__float2int_rn(acc[0][r]) << 24) + ((long long)__float2int_rn(acc[1][r]) << 16) +
                 ((long long)__float2int_rn(acc[2][r]) << 8) + (long long)__float2int_rn(acc[3][r]);
        lo[r] += ((long long)__float2int_rn(acc[4][r]) << 24) + ((long long)__float2int_rn(acc[5][r]) << 16) +
                 ((long long)__float2int_rn(acc[6][r]) << 8) + (long long)__float2int_rn(acc[7][r]);
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      // element (m0 + g + 8 (r / 2), n0 + 2 t + r % 2): the sums of digit
      // order 7 carry the weight 2^{56 + 56 - 56} of the scaled integers
      const int i = m0 + g + 8 * (r >> 1), j = n0 + 2 * t + (r & 1);
      if (i < M && j < Nn) {
        const int e = ea(i) + eb(j);
        const double v = e >= kDigitBad / 4 ? __longlong_as_double(0x7ff8000000000000ll)
                         : e < kDigitNone / 2 ? 0.0 : digit_value(hi[r], lo[r], e - 68);
        epi(i, j, v);
      }
    }
  }
}

// largest digit exponent over the CTA (collective; red: one int per warp)
static __device__ __forceinline__ int digit_cta_max(int e, int* red) {
  e = __reduce_max_sync(0xffffffffu, e);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = e;
  __syncthreads();
  int m = red[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) m = max(m, red[w]);
  return m;
}

}  // namespace pqmc
