// Products of FP64 and FP32 matrices on the 16-bit tensor cores, exact up to a chosen truncation
// (the error-free splitting of Ozaki, Ogita, Oishi and Rump 2012, in the tensor-core form of Mukunoki,
// Ozaki, Ogita and Imamura 2020): each operand becomes a fixed-point integer relative to the scale of its row (left
// operand) or column (right operand), written as ND balanced digits d_0 (most significant) .. d_{ND-1} of BD bits; every digit is
// an exact fp16 number, and the products of two digits summed over K stay below 2^24, so the FP32
// accumulators of mma.sync hold them exactly.  Digit products of one order i + j share an
// accumulator; orders above NO - 1 are dropped.
//   FP64: 7 digits of 8 bits, orders 0..7:  34 digit products, 7 x K x 2^14 < 2^24 for K <= 146
//   FP32: 3 digits (9, 9 and up to 11 bits), orders 0..2: 6 digit products; orders 0 and 1 are exact sums,
//         2 x K x 2^16 < 2^24 for K <= 127
//
// Why on this GPU: the FP64 pipe gives 2 multiply-adds a clock and SM (DFMA measured at 588 G/s; one
// warp instruction occupies a sub-partition's pipe for 64 clocks), mma.sync with fp16 operands 1,032.
// 34 digit products per FP64 product (7 digits, orders 0..7) are 15 times cheaper than the DFMAs they replace.
// FP32: 6 digit products cost 0.75 of the FFMA time at peak rates, leave the CUDA cores to the tanh and need no
// register tiles of weights.
//
// Error: relative to the largest element of the row times the largest of the column, 2^-28 (FP32) or 2^-54 (FP64)
// a term, where FMAs round every partial sum.  On nets whose columns are alike (kSpread) energies and
// forces are as close to FP64 as with FMAs or closer: over 22 nets (scaled by 0.01 to 40, uneven rows and columns, heavy
// tails, no biases) the ratio of the errors is 0.3 to 1.05 in FP32, 0.8 to 1.14 in FP64.
#pragma once

#include "common.cuh"

namespace dpg {
namespace dig {

// Largest ratio of a column's largest weight to the rms of its other nonzero weights that the digit products take.
// All of a column is cut relative to its largest weight, and that one's input may be zero (a large weight saturates
// its unit, whose gradient vanishes), so the others must keep their bits beside it: at 10 their cuts are 2^-52.5 (FP64)
// of them, the error of the FMAs.  Normal weights reach 5.  Nets with more spread take the plain kernels (simt.cu).
constexpr float kSpread = 10.f;

template <class T> struct Fmt;
template <> struct Fmt<double> {
  static constexpr int BD = 8, ND = 7, NO = 8;  // bits a digit, digits, product orders kept
  using V = long long;                  // fixed point, 54 fraction bits (activations)
};
template <> struct Fmt<float> {
  static constexpr int BD = 9, ND = 3, NO = 3;
  using V = float;
};

// uint4 loads per lane and fragment set: digits 2q and 2q + 1 of a B fragment in one 16-byte word.
template <class T> struct Frag {
  static constexpr int Q = (Fmt<T>::ND + 1) / 2;
};

// (not volatile: independent products may be interleaved)
__device__ __forceinline__ void hmma16(float* c, const uint4& a, uint32_t b0, uint32_t b1) {
  asm(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void hmma8(float* c, uint32_t a0, uint32_t a1, uint32_t b0) {
  asm(
      "mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

// The same with a zero accumulator (no registers to clear first).
__device__ __forceinline__ void hmma16z(float* c, const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1), "f"(0.f));
}

// Two bytes u0 (digit + 128 of the even column) and u1 (odd column) as a half2 of the digits:
// 0x6400 | u is 1024 + u in fp16, and 1024 + 128 is taken off exactly.
__device__ __forceinline__ uint32_t bytes_to_half2(uint32_t both) {
  const uint32_t h = (both & 0x00ff00ffu) | 0x64006400u;
  const __half2 d = __hsub2(*reinterpret_cast<const __half2*>(&h), __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480)));
  return *reinterpret_cast<const uint32_t*>(&d);
}

// The digits, each made non-negative, of a fixed-point value |v| <= 2^(BD ND - 2).
__device__ __forceinline__ unsigned long long biased(long long v) {
  return (unsigned long long)v + 0x0080808080808080ull;
}
// out[i] = half2 of digit i of (u0, u1).
__device__ __forceinline__ void split2(unsigned long long u0, unsigned long long u1, uint32_t* out) {
  const uint32_t l0 = (uint32_t)u0, h0 = (uint32_t)(u0 >> 32), l1 = (uint32_t)u1, h1 = (uint32_t)(u1 >> 32);
  // byte b of word 0 to byte 0, byte b of word 1 to byte 2
  out[0] = bytes_to_half2(__byte_perm(h0, h1, 0x0602));
  out[1] = bytes_to_half2(__byte_perm(h0, h1, 0x0501));
  out[2] = bytes_to_half2(__byte_perm(h0, h1, 0x0400));
  out[3] = bytes_to_half2(__byte_perm(l0, l1, 0x0703));
  out[4] = bytes_to_half2(__byte_perm(l0, l1, 0x0602));
  out[5] = bytes_to_half2(__byte_perm(l0, l1, 0x0501));
  out[6] = bytes_to_half2(__byte_perm(l0, l1, 0x0400));
}
// FP32: |x| <= 256 as three fp16 numbers that carry their own weights: the nearest integer, the nearest multiple of 2^-9 of
// what is left (nine bits each, by adding and subtracting 1.5 x 2^23 times the step), and the rest, which is
// below 2^-10 and kept within 2^-22.  Five additions a value, where integer digits took ten instructions.
__device__ __forceinline__ void split2f(float x0, float x1, uint32_t* out) {
  constexpr float m0 = 12582912.f, m1 = m0 / 512.f;
  const float a0 = __fsub_rn(__fadd_rn(x0, m0), m0), a1 = __fsub_rn(__fadd_rn(x1, m0), m0);
  const float r0 = __fsub_rn(x0, a0), r1 = __fsub_rn(x1, a1);
  const float b0 = __fsub_rn(__fadd_rn(r0, m1), m1), b1 = __fsub_rn(__fadd_rn(r1, m1), m1);
  const __half2 h0 = __floats2half2_rn(a0, a1), h1 = __floats2half2_rn(b0, b1),
                h2 = __floats2half2_rn(__fsub_rn(r0, b0), __fsub_rn(r1, b1));
  out[0] = *reinterpret_cast<const uint32_t*>(&h0);
  out[1] = *reinterpret_cast<const uint32_t*>(&h1);
  out[2] = *reinterpret_cast<const uint32_t*>(&h2);
}

// All kept digit products of one (16 x 16) x (16 x 8) block: consecutive instructions go to different
// accumulators.
// FIRST: the block's first product of each order overwrites the accumulator.
template <class T, bool FIRST = false>
__device__ __forceinline__ void block16(float (*acc)[4], const uint4* a, const uint4* b) {
  constexpr int ND = Fmt<T>::ND, NO = Fmt<T>::NO;
#pragma unroll
  for (int j = 0; j < ND; ++j) {
    const uint32_t b0 = (j & 1) ? b[j >> 1].z : b[j >> 1].x, b1 = (j & 1) ? b[j >> 1].w : b[j >> 1].y;
#pragma unroll
    for (int i = 0; i < ND; ++i)
      if (i + j < NO) {
        if (FIRST && (j == 0 || i == ND - 1)) hmma16z(acc[i + j], a[i], b0, b1);
        else hmma16(acc[i + j], a[i], b0, b1);
      }
  }
}
template <class T>
__device__ __forceinline__ void block8(float (*acc)[4], const uint2* a, const uint4* b) {
  constexpr int ND = Fmt<T>::ND, NO = Fmt<T>::NO;
#pragma unroll
  for (int j = 0; j < ND; ++j) {
    const uint32_t b0 = (j & 1) ? b[j >> 1].z : b[j >> 1].x;
#pragma unroll
    for (int i = 0; i < ND; ++i)
      if (i + j < NO) hmma8(acc[i + j], a[i].x, a[i].y, b0);
  }
}

template <class T>
__device__ __forceinline__ void zero_acc(float (*acc)[4]) {
#pragma unroll
  for (int o = 0; o < Fmt<T>::NO; ++o)
#pragma unroll
    for (int e = 0; e < 4; ++e) acc[o][e] = 0.f;
}

// The accumulators of one output (element e of the fragment) as two integers: orders 0..3 in units of
// 256^(2 (ND - 1) - 3), orders 4..7 in units of 256^(2 (ND - 1) - 7).  |orders| < 2^24.
struct Pair64 {
  long long hi, lo;
};
__device__ __forceinline__ long long join4(float a0, float a1, float a2, float a3) {
  const long long t = (long long)__float2int_rn(a0) * 256 + __float2int_rn(a1);
  const long long u = (long long)__float2int_rn(a2) * 256 + __float2int_rn(a3);
  return (t << 16) + u;
}
__device__ __forceinline__ Pair64 join(const float (*acc)[4], int e) {
  Pair64 p;
  p.hi = join4(acc[0][e], acc[1][e], acc[2][e], acc[3][e]);
  p.lo = join4(acc[4][e], acc[5][e], acc[6][e], acc[7][e]);
  return p;
}
// FP32: sum of the orders (the digits carry their weights).
__device__ __forceinline__ float join_f(const float (*acc)[4], int e) { return acc[0][e] + (acc[1][e] + acc[2][e]); }

// 2^e as FP64 / FP32 (normal range).
__host__ __device__ __forceinline__ double pow2d(int e) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)(1023 + e) << 52);
#else
  return std::ldexp(1.0, e);
#endif
}

// tanh of a fixed-point argument (zs fraction bits, 40 <= zs <= 56) as a fixed-point value with 54
// fraction bits, in integer arithmetic: the tanh of CUDA's library costs 17 to 38 FP64 operations and
// the FP64 pipe is this path's scarcest unit, 32 integer instructions fit in one FP64 instruction's slot.
// Taylor polynomial of degree 6 about the nearest multiple of 1/64 (degree 7 economised), the
// leading coefficients in 64 bits, the rest in 32; beyond 20 the result is 1.  Error
// against the exact value: rms 2^-55.2, at most 2^-52.4 (5,200 arguments over all intervals, tests/test_tanh_fixed.py).
constexpr int kTanhN = 1281;
struct TanhTab {
  longlong2 a[kTanhN];  // c0, c1 (62 fraction bits)
  int4 b[kTanhN];       // c2 (62 fraction bits, two words), c3 (32 fraction bits), c4 (FP32)
  float2 c[kTanhN];     // c5, c6
};

__device__ __forceinline__ long long tanh_fixed(long long z, int zs, const TanhTab* tab) {
  const long long lim = 32ll << zs;
  z = z > lim ? lim : (z < -lim ? -lim : z);
  const bool neg = z < 0;
  const long long a = neg ? -z : z;
  int k = (int)((a + (1ll << (zs - 7))) >> (zs - 6));
  long long d = a - ((long long)k << (zs - 6));
  if (k >= kTanhN - 1) {
    k = kTanhN - 1;
    d = 0;
  }
  const long long D = d << (70 - zs);
  const int Dh = (int)(D >> 32);
  const longlong2 ca = tab->a[k];
  const int4 cb = tab->b[k];
  const float2 cc = tab->c[k];
  const float df = (float)Dh * 3.637978807091713e-12f;  // 2^-38
  const float F = fmaf(df, fmaf(df, cc.y, cc.x), __int_as_float(cb.w));
  const int u3 = cb.z + __float2int_rn(df * F * 4294967296.f);
  const long long c2 = ((long long)cb.y << 32) | (unsigned)cb.x;
  const long long u2 = c2 + (((long long)Dh * u3) >> 8);
  const long long u1 = ca.y + (__mul64hi(D, u2) >> 6);
  long long t = ca.x + (__mul64hi(D, u1) >> 6);
  t = (t + 128) >> 8;
  return neg ? -t : t;
}

}  // namespace dig
}  // namespace dpg
