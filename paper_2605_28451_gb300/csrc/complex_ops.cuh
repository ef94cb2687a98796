// Complex arithmetic and small DFT blocks for the register-resident butterflies.
//
// All arithmetic is FP32 (float2 = re, im), whatever the storage type: the
// paper's FP16-storage / FP32-compute mode (Section VI), which keeps every
// multiply-add of a butterfly in FP32 registers and rounds to FP16 only where
// data leaves the chip.
//
// The blocks compute the forward DFT  X[k] = sum_r v[r] exp(-2 pi i r k / R)
// for R = 2, 4, 8, 16, 32, 64, in natural output order.  The inverse is never needed:
// the inverse transform is realised as conj(FFT(conj z)) (Section III-B).
#pragma once

#include <cuda_runtime.h>

namespace bfp {

// Packed FP32 (sm_100-family f32x2): one instruction adds or subtracts both
// components of a complex value held as a 64-bit register pair.
#ifndef BFP_F32X2
#define BFP_F32X2 1
#endif

__device__ __forceinline__ unsigned long long as_u64(float2 a) { return *reinterpret_cast<unsigned long long*>(&a); }
__device__ __forceinline__ float2 as_f2(unsigned long long u) { return *reinterpret_cast<float2*>(&u); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) {
#if BFP_F32X2
  unsigned long long r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(b)));
  return as_f2(r);
#else
  return make_float2(a.x + b.x, a.y + b.y);
#endif
}
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
#if BFP_F32X2
  unsigned long long r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(b)));
  return as_f2(r);
#else
  return make_float2(a.x - b.x, a.y - b.y);
#endif
}
// Both components times the same real factor.
__device__ __forceinline__ float2 cmul_real2(float2 a, float s) {
#if BFP_F32X2
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(make_float2(s, s))));
  return as_f2(r);
#else
  return make_float2(a.x * s, a.y * s);
#endif
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
// (a.x, a.y) * (s.x, s.y), component by component.
__device__ __forceinline__ float2 cmul_parts(float2 a, float2 s) {
#if BFP_F32X2
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(as_u64(a)), "l"(as_u64(s)));
  return as_f2(r);
#else
  return make_float2(a.x * s.x, a.y * s.y);
#endif
}
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// multiply by -i
__device__ __forceinline__ float2 cmul_mi(float2 a) { return make_float2(a.y, -a.x); }

// Constant twiddles of the 16-point block, W16^e = exp(-2 pi i e / 16).
constexpr float kC1 = 0.92387953251128675613f;   // cos(pi/8)
constexpr float kS1 = 0.38268343236508977173f;   // sin(pi/8)
constexpr float kR2 = 0.70710678118654752440f;   // sqrt(1/2)

// (x + iy) * W16^2 = sqrt(1/2) * ((x + y) + i (y - x))
__device__ __forceinline__ float2 mul_w16_2(float2 a) { return cmul_real2(make_float2(a.x + a.y, a.y - a.x), kR2); }
// (x + iy) * W16^6 = sqrt(1/2) * ((y - x) - i (x + y))
__device__ __forceinline__ float2 mul_w16_6(float2 a) { return cmul_real2(make_float2(a.y - a.x, -a.x - a.y), kR2); }
__device__ __forceinline__ float2 mul_w16_1(float2 a) { return cmul(a, make_float2(kC1, -kS1)); }
__device__ __forceinline__ float2 mul_w16_3(float2 a) { return cmul(a, make_float2(kS1, -kC1)); }
__device__ __forceinline__ float2 mul_w16_9(float2 a) { return cmul(a, make_float2(-kC1, kS1)); }

// 4-point forward DFT in place: (a0, a1, a2, a3) -> (X0, X1, X2, X3).
// e = -i (a1 - a3) is formed with two scalar subtractions straight into the
// swapped order, so every other step is one packed add or subtract.
__device__ __forceinline__ void dft4(float2& a0, float2& a1, float2& a2, float2& a3) {
  const float2 t0 = cadd(a0, a2), t1 = csub(a0, a2);
  const float2 t2 = cadd(a1, a3);
  const float2 e = make_float2(a1.y - a3.y, a3.x - a1.x);
  a0 = cadd(t0, t2);
  a2 = csub(t0, t2);
  a1 = cadd(t1, e);
  a3 = csub(t1, e);
}

template <int R, bool FINE = false> struct Dft;

template <bool FINE> struct Dft<2, FINE> {
  __device__ __forceinline__ static void run(float2 (&v)[2]) {
    const float2 a = v[0], b = v[1];
    v[0] = cadd(a, b);
    v[1] = csub(a, b);
  }
};

template <bool FINE> struct Dft<4, FINE> {
  __device__ __forceinline__ static void run(float2 (&v)[4]) { dft4(v[0], v[1], v[2], v[3]); }
};

// a + sqrt(1/2) b and a - sqrt(1/2) b, one packed FMA each: the eighth roots'
// common factor rides on the butterfly that follows instead of a multiply.
__device__ __forceinline__ float2 add_r2(float2 a, float2 b) {
#if BFP_F32X2
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(as_u64(b)), "l"(as_u64(make_float2(kR2, kR2))), "l"(as_u64(a)));
  return as_f2(r);
#else
  return make_float2(fmaf(b.x, kR2, a.x), fmaf(b.y, kR2, a.y));
#endif
}
__device__ __forceinline__ float2 sub_r2(float2 a, float2 b) {
#if BFP_F32X2
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(as_u64(b)), "l"(as_u64(make_float2(-kR2, -kR2))), "l"(as_u64(a)));
  return as_f2(r);
#else
  return make_float2(fmaf(b.x, -kR2, a.x), fmaf(b.y, -kR2, a.y));
#endif
}

// 8 = 2 x 4: r = r1 + 2 r2, k = k2 + 4 k1.  The odd half's W8 and W8^3 have
// their sqrt(1/2) folded into the last butterflies.
template <bool FINE> struct Dft<8, FINE> {
  __device__ __forceinline__ static void run(float2 (&v)[8]) {
    dft4(v[0], v[2], v[4], v[6]);           // r1 = 0 -> a0[k2] at v[0,2,4,6]
    dft4(v[1], v[3], v[5], v[7]);           // r1 = 1 -> a1[k2] at v[1,3,5,7]
    const float2 s1 = make_float2(v[3].x + v[3].y, v[3].y - v[3].x);      // sqrt(2) W8 a1[1]
    const float2 s3 = make_float2(v[7].y - v[7].x, -v[7].x - v[7].y);     // sqrt(2) W8^3 a1[3]
    const float2 m = cmul_mi(v[5]);
    const float2 o[8] = {cadd(v[0], v[1]), add_r2(v[2], s1), cadd(v[4], m), add_r2(v[6], s3),
                         csub(v[0], v[1]), sub_r2(v[2], s1), csub(v[4], m), sub_r2(v[6], s3)};
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = o[i];
  }
};

// 16 = 4 x 4: r = r1 + 4 r2, k = k2 + 4 k1.
template <bool FINE> struct Dft<16, FINE> {
  __device__ __forceinline__ static void run(float2 (&v)[16]) {
#pragma unroll
    for (int r1 = 0; r1 < 4; ++r1) dft4(v[r1], v[r1 + 4], v[r1 + 8], v[r1 + 12]);
    // a[r1][k2] sits at v[r1 + 4 k2]; multiply by W16^(r1 k2).
    v[5] = mul_w16_1(v[5]);
    v[9] = mul_w16_2(v[9]);
    v[13] = mul_w16_3(v[13]);
    v[6] = mul_w16_2(v[6]);
    v[10] = cmul_mi(v[10]);
    v[14] = mul_w16_6(v[14]);
    v[7] = mul_w16_3(v[7]);
    v[11] = mul_w16_6(v[11]);
    v[15] = mul_w16_9(v[15]);
    // DFT-4 over r1 for each k2; X[k2 + 4 k1] = result k1.
    float2 o[16];
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
      float2 a0 = v[4 * k2 + 0], a1 = v[4 * k2 + 1], a2 = v[4 * k2 + 2], a3 = v[4 * k2 + 3];
      dft4(a0, a1, a2, a3);
      o[k2] = a0;
      o[k2 + 4] = a1;
      o[k2 + 8] = a2;
      o[k2 + 12] = a3;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = o[i];
  }
};

// Roots of unity as compile-time constants: cos and sin of an exact dyadic
// fraction of a turn, from the Taylor series in FP64 on [0, pi / 4] and the
// circle's symmetries, rounded once to FP32.
__host__ __device__ constexpr double taylor_cos(double x) {
  double t = 1.0, s = 1.0;
  for (int k = 1; k <= 12; ++k) {
    t *= -x * x / double((2 * k - 1) * (2 * k));
    s += t;
  }
  return s;
}
__host__ __device__ constexpr double taylor_sin(double x) {
  double t = x, s = x;
  for (int k = 1; k <= 12; ++k) {
    t *= -x * x / double((2 * k) * (2 * k + 1));
    s += t;
  }
  return s;
}
// cos(2 pi e / m), 0 <= e < m, m a multiple of 8.
__host__ __device__ constexpr double cos_turn(int e, int m) {
  if (2 * e > m) e = m - e;                                    // cos(-x) = cos x
  if (4 * e > m) return -cos_turn(m / 2 - e, m);               // cos(pi - x) = -cos x
  const double turn = 6.28318530717958647692528676655900577;
  return 8 * e <= m ? taylor_cos(turn * e / m) : taylor_sin(turn * (m / 4 - e) / m);
}
__host__ __device__ constexpr double sin_turn(int e, int m) { return cos_turn((e + 3 * m / 4) % m, m); }   // cos(x - pi / 2)

// a * W_M^E = a * exp(-2 pi i E / M); the eighth roots cost two to four
// instructions less than a full product.  cos(pi / 16) and cos(pi / 8) happen to
// lie almost half an FP32 step (0.499 and 0.475) from their rounded values, and
// every line takes the same few constants, so their errors add up: FINE, for
// results stored in FP32, adds the low part of the constant that is further off,
// at two multiplies a product.  Relative L2 error of FP32 lines in passes of radix
// 16, in these radices without the low parts, and with them (1e-7): 1024 points
// 1.083, 1.107, 1.031; 16384 1.326, 1.351, 1.267; 32768 1.378, 1.431, 1.354;
// 65536 1.449, 1.473, 1.402.  It costs 1 to 2 % of the time from 8192 points on
// (2^26 points: 16384 221.6 -> 223.9 us, 65536 251.5 -> 257.6), none below.
template <int E, int M, bool FINE>
__device__ __forceinline__ float2 mul_root(float2 a) {
  constexpr int e = E % M;
  if constexpr (e == 0) return a;
  else if constexpr (4 * e == M) return cmul_mi(a);
  else if constexpr (8 * e == M) return mul_w16_2(a);
  else if constexpr (8 * e == 3 * M) return mul_w16_6(a);
  else {
    constexpr double cd = cos_turn(e, M), sd = -sin_turn(e, M);
    constexpr float c = float(cd), s = float(sd), cl = float(cd - double(c)), sl = float(sd - double(s));
    if constexpr (!FINE) return cmul(a, make_float2(c, s));
    else if constexpr (cl * cl >= sl * sl)
      return make_float2(fmaf(a.x, c, fmaf(-a.y, s, a.x * cl)), fmaf(a.x, s, fmaf(a.y, c, a.y * cl)));
    else
      return make_float2(fmaf(a.x, c, fmaf(-a.y, s, -a.y * sl)), fmaf(a.x, s, fmaf(a.y, c, a.x * sl)));
  }
}

// v[k2] *= W_M^(R1 k2) for the eight k2.
template <int R1, int M, bool FINE>
__device__ __forceinline__ void mul_roots8(float2 (&v)[8]) {
  v[1] = mul_root<R1, M, FINE>(v[1]);
  v[2] = mul_root<2 * R1, M, FINE>(v[2]);
  v[3] = mul_root<3 * R1, M, FINE>(v[3]);
  v[4] = mul_root<4 * R1, M, FINE>(v[4]);
  v[5] = mul_root<5 * R1, M, FINE>(v[5]);
  v[6] = mul_root<6 * R1, M, FINE>(v[6]);
  v[7] = mul_root<7 * R1, M, FINE>(v[7]);
}

// Column r1 of an R1 x 8 split: the 8-point DFT of v[r1 + R1 r2] over r2,
// times W_M^(r1 k2), back in place at v[r1 + R1 k2].
template <int r1, int R1, bool FINE, int M>
__device__ __forceinline__ void dft8_column(float2 (&v)[M]) {
  float2 u[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) u[i] = v[r1 + R1 * i];
  Dft<8>::run(u);
  mul_roots8<r1, M, FINE>(u);
#pragma unroll
  for (int i = 0; i < 8; ++i) v[r1 + R1 * i] = u[i];
}

// 32 = 4 x 8: r = r1 + 4 r2, k = k2 + 8 k1.
template <bool FINE> struct Dft<32, FINE> {
  __device__ __forceinline__ static void run(float2 (&v)[32]) {
    dft8_column<0, 4, FINE>(v);
    dft8_column<1, 4, FINE>(v);
    dft8_column<2, 4, FINE>(v);
    dft8_column<3, 4, FINE>(v);
    float2 o[32];
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) {
      float2 a0 = v[4 * k2], a1 = v[4 * k2 + 1], a2 = v[4 * k2 + 2], a3 = v[4 * k2 + 3];
      dft4(a0, a1, a2, a3);
      o[k2] = a0;
      o[k2 + 8] = a1;
      o[k2 + 16] = a2;
      o[k2 + 24] = a3;
    }
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = o[i];
  }
};

// 64 = 8 x 8: r = r1 + 8 r2, k = k2 + 8 k1.
template <bool FINE> struct Dft<64, FINE> {
  __device__ __forceinline__ static void run(float2 (&v)[64]) {
    dft8_column<0, 8, FINE>(v);
    dft8_column<1, 8, FINE>(v);
    dft8_column<2, 8, FINE>(v);
    dft8_column<3, 8, FINE>(v);
    dft8_column<4, 8, FINE>(v);
    dft8_column<5, 8, FINE>(v);
    dft8_column<6, 8, FINE>(v);
    dft8_column<7, 8, FINE>(v);
    float2 o[64];
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) {
      float2 u[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) u[i] = v[8 * k2 + i];
      Dft<8>::run(u);
#pragma unroll
      for (int i = 0; i < 8; ++i) o[k2 + 8 * i] = u[i];
    }
#pragma unroll
    for (int i = 0; i < 64; ++i) v[i] = o[i];
  }
};

}  // namespace bfp
