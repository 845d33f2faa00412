// Rank-16 updates of FP64 and FP32-pair matrices on the tensor cores: C += sum_{q<16} x_q y_q^T, by
// exact slicing (Ozaki et al., Numer. Algorithms 2012). Each row's 16 x and each column's 16 y, scaled
// by a power of two, are cut into 6 balanced digits of 10 bits (|d| <= 512, exact in FP16); the 21 digit
// products s + t <= 5 accumulate in six FP32 groups g = s + t by mma.sync, exact for g <= 3
// (16 * 4 * 2^18 = 2^24). What is dropped is below 2^-57 (FP64; 2^-54 for FP32 pairs) of the product of
// the row's and the column's maxima. tcgen05 would need 128 rows per tile and TMEM round trips for one
// k-step; mma.sync issues from the registers at hand.
#pragma once
#include <cuda_fp16.h>

#include <cstring>

#include "df.cuh"

namespace nmc {
namespace {

constexpr int kFoldK = 16;
constexpr int kFDig = 6, kFW = 10, kFBits = 59;

// How a value's digits are cut
template <typename T> struct Digits;
template <> struct Digits<df2> {
  // biased exponent of |a|
  static __device__ __forceinline__ int expo(df2 a) { return (__float_as_int(a.hi) >> 23) & 0xff; }
  static constexpr int kExpMin = 9, kExpMax = 0xff;
  // The terms of two k as FP16 digit pairs, most significant first. A term in units of 2^(E - 135)
  // is below 512; adding kM 2^(-10 s) (ulp 2^(-10 s)) rounds it to its digit s, which then stands in
  // the low mantissa bits on top of 0x6600, FP16's 1536. The low part joins after the first digit by
  // exact sums (Fast2Sum: what is left of the high part is 0 or at least twice as large), its rest
  // after the second and the third, so that no digit exceeds 512: beyond, FP16's steps are 2.
  static __device__ __forceinline__ void digits(df2 a, df2 b, int E, unsigned (&w)[kFDig]) {
    const float sc = __int_as_float((262 - E) << 23);
    unsigned t0[kFDig], t1[kFDig];
    split(a, sc, t0);
    split(b, sc, t1);
#pragma unroll
    for (int s = 0; s < kFDig; ++s) w[s] = __byte_perm(t0[s], t1[s], 0x5410);
  }
  static __device__ __forceinline__ void split(df2 a, float sc, unsigned (&t)[kFDig]) {
    float v = __fmul_rn(a.hi, sc), e = __fmul_rn(a.lo, sc), m = __int_as_float(0x4b406600);
#pragma unroll
    for (int s = 0; s < kFDig; ++s) {
      if (s == 1 || s == 2) {
        const float q = __fadd_rn(v, e);
        e = __fsub_rn(e, __fsub_rn(q, v));
        v = q;
      }
      if (s == 3) v = __fadd_rn(v, e);
      const float x = __fadd_rn(v, m);
      t[s] = __float_as_uint(x);
      v = __fsub_rn(v, __fsub_rn(x, m));
      m *= 0x1p-10f;
    }
  }
  // what a row's (column's) digit sums are multiplied by: 2^(E - 135), or NaN where a term is not finite
  static __device__ __forceinline__ int scale(int E) {
    return E == kExpMax ? 0x7fc00000 : (E - 8) << 23;
  }
};
template <> struct Digits<double> {
  static __device__ __forceinline__ int expo(double a) { return (__double2hiint(a) >> 20) & 0x7ff; }
  static __device__ __forceinline__ long long fixed(double a, int E) {
    const unsigned h = (unsigned)__double2hiint(a), l = (unsigned)__double2loint(a);
    const int e = (int)((h >> 20) & 0x7ffu);
    const unsigned long long m =
        ((unsigned long long)(__funnelshift_l(l, h, 11) | 0x80000000u) << 32 | (l << 11));
    const long long v = e == 0 ? 0ll : (long long)(m >> min(64 - kFBits + E - e, 63));
    return (int)h < 0 ? -v : v;
  }
  static constexpr int kExpMin = 1, kExpMax = 0x7ff;
  // Adding 512 to every 10-bit field of the term in units of 2^(E - 1022 - kFBits) and reading the
  // fields less 512 gives balanced digits; a field added to 0x6400, FP16's 1024, is 1536 + digit.
  static __device__ __forceinline__ void digits(double a, double b, int E, unsigned (&w)[kFDig]) {
    const unsigned long long u0 = (unsigned long long)(fixed(a, E) + 0x0802008020080200ll);
    const unsigned long long u1 = (unsigned long long)(fixed(b, E) + 0x0802008020080200ll);
#pragma unroll
    for (int s = 0; s < kFDig; ++s) {
      const int bit = kFW * (kFDig - 1 - s);
      w[s] = __byte_perm((unsigned)(u0 >> bit), (unsigned)(u1 >> bit), 0x5410);
      if (s > 0) w[s] &= 0x03ff03ffu;   // (the first digit's field may reach 1024)
      w[s] += 0x64006400u;
    }
  }
  static __device__ __forceinline__ int scale(int E) { return E; }
};

// byte offset of the 16-byte half h (k = 8 h ..) of a digit row r: rows of 32 bytes, the halves
// exchanged in every second group of four rows so that ldmatrix meets all banks
__device__ __forceinline__ int digit_off(int r, int h) { return r * 32 + ((h ^ ((r >> 2) & 1)) << 4); }

// Cut the 16 terms of one row (or column) into digits, most significant first: store(s, h, .) takes
// half h of digit s
template <typename T, typename F>
__device__ __forceinline__ void cut16_to(const T (&x)[kFoldK], int E, F store) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    unsigned w[4][kFDig];
#pragma unroll
    for (int i = 0; i < 4; ++i) Digits<T>::digits(x[8 * h + 2 * i], x[8 * h + 2 * i + 1], E, w[i]);
#pragma unroll
    for (int s = 0; s < kFDig; ++s) {
      unsigned d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const __half2 v = __hadd2(*reinterpret_cast<__half2*>(&w[i][s]), __float2half2_rn(-1536.f));
        d[i] = *reinterpret_cast<const unsigned*>(&v);
      }
      store(s, h, make_uint4(d[0], d[1], d[2], d[3]));
    }
  }
}
// to row r at dst, `stride` bytes apart
template <typename T>
__device__ __forceinline__ void cut16(const T (&x)[kFoldK], int E, unsigned char* dst, int r, int stride) {
  cut16_to(x, E, [&](int s, int h, uint4 v) { *reinterpret_cast<uint4*>(dst + s * stride + digit_off(r, h)) = v; });
}

__device__ __forceinline__ void ldm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_h(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// One entry of G plus its digit sums sum_g a_g 2^(-10 g) times the row's and the column's scale.
// a_0 + a_1 2^-10 + a_2 2^-20 as an exact pair by Fast2Sum: where the smaller-magnitude operand comes
// first, the sum is short enough to be exact (a_0 is an integer, |a_1 2^-10| < 2^13, |a_2 2^-20| < 13).
__device__ __forceinline__ void fold_entry(df2& G, const float (&a)[kFDig], int ea, int eb) {
  const float s = __fmaf_rn(a[1], 0x1p-10f, a[0]);
  const float e1 = __fmaf_rn(a[1], 0x1p-10f, -__fsub_rn(s, a[0]));
  const float h = __fmaf_rn(a[2], 0x1p-20f, s);
  const float e2 = __fmaf_rn(a[2], 0x1p-20f, -__fsub_rn(h, s));
  float l = __fmaf_rn(a[3], 0x1p-30f, __fadd_rn(e1, e2));
  l = __fmaf_rn(a[5], 0x1p-50f, __fmaf_rn(a[4], 0x1p-40f, l));
  const float sc = __fmul_rn(__int_as_float(ea), __int_as_float(eb));
  const float th = __fmul_rn(h, sc), q = __fadd_rn(G.hi, th), b = __fsub_rn(q, G.hi);
  const float e = __fadd_rn(__fsub_rn(G.hi, __fsub_rn(q, b)), __fsub_rn(th, b));
  G = df_norm(q, __fadd_rn(e, __fmaf_rn(l, sc, G.lo)));
}
__device__ __forceinline__ void fold_entry(double& G, const float (&a)[kFDig], int ea, int eb) {
  if (max(ea, eb) >= Digits<double>::kExpMax) {   // an infinity or a NaN among the terms
    G = __longlong_as_double(0x7ff8000000000000ll);
    return;
  }
  int q[kFDig];
#pragma unroll
  for (int s = 0; s < kFDig; ++s) q[s] = __float2int_rn(a[s]);
  long long H = (long long)q[0] * (1 << 20) + ((long long)q[1] * (1 << 10) + q[2]);
  long long L = (long long)q[3] * (1 << 20) + ((long long)q[4] * (1 << 10) + q[5]);
  H += L >> 30;   // (H 2^30 + L) 2^-50
  L &= (1ll << 30) - 1;
  const int s = min(__clzll(H ^ (H >> 63)) - 1, 30);
  const long long v = (H << s) + (L >> (30 - s));
  if (v == 0) return;
  // to FP64 in integers (a conversion would take the FP64 pipe as long as the addition below does)
  const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll(m), k = ea + eb - 2 * 1022 - 18 - 20 - s, e = k - z + 1086;
  const unsigned long long t = m << z, f = (t >> 11) + ((t >> 10) & 1);
  const unsigned long long b = ((unsigned long long)(unsigned)(e - 1) << 52) + f;
  G += e >= 1 && e <= 2045 ? __longlong_as_double((long long)(b | ((unsigned long long)v & (1ull << 63))))
                           : ldexp((double)v, k);
}

// C(r, c) += sum_q x_q[r] y_q[c] for nrows x ncols entries, 16 x 16 blocks shared out to the warps.
// row(r): pointer to C's row r; pair: rows 16-byte aligned and ncols even. xd, yd: shared addresses of the digits,
// xs, ys bytes from digit to digit; xe, ye: scales of rows and columns.
template <typename T, typename Row>
__device__ __forceinline__ void fold_tiles(Row row, unsigned xd, int xs, const int* xe, unsigned yd, int ys,
                                           const int* ye, int nrows, int ncols, bool pair, int warp,
                                           int nwarps) {
  const int lane = threadIdx.x & 31;
  const int nr = (nrows + 15) >> 4, nc = (ncols + 15) >> 4, per = (nr * nc + nwarps - 1) / nwarps;
  const int ar = lane & 15, ah = lane >> 4;                             // ldmatrix rows, halves
  const int br = (lane & 7) + ((lane >> 4) & 1) * 8, bh = (lane >> 3) & 1;
  for (int job = warp * per; job < min((warp + 1) * per, nr * nc); ++job) {
    const int rb = job / nc * 16, cb = job % nc * 16;
    float acc[2][4][kFDig];
#pragma unroll
    for (int n2 = 0; n2 < 2; ++n2)
#pragma unroll
      for (int w = 0; w < 4; ++w)
#pragma unroll
        for (int g = 0; g < kFDig; ++g) acc[n2][w][g] = 0.f;
    float4 c4[2][2];   // C's entries, two each
#pragma unroll
    for (int n2 = 0; n2 < 2; ++n2)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = rb + (lane >> 2) + 8 * h, cc = cb + 8 * n2 + 2 * (lane & 3);
        if (r >= nrows || cc >= ncols) continue;
        const T* p = row(r) + cc;
        if (pair) {
          c4[n2][h] = *(const float4*)p;
        } else {
          const T v[2] = {p[0], p[cc + 1 < ncols ? 1 : 0]};
          memcpy(&c4[n2][h], v, sizeof v);
        }
      }
    unsigned bf[kFDig][4];
#pragma unroll
    for (int s = 0; s < kFDig; ++s) ldm4(bf[s], yd + s * ys + digit_off(cb + br, bh));
#pragma unroll
    for (int s = 0; s < kFDig; ++s) {
      unsigned af[4];
      ldm4(af, xd + s * xs + digit_off(rb + ar, ah));
#pragma unroll
      for (int q = 0; q + s < kFDig; ++q)
#pragma unroll
        for (int n2 = 0; n2 < 2; ++n2) {
          float d[4] = {acc[n2][0][s + q], acc[n2][1][s + q], acc[n2][2][s + q], acc[n2][3][s + q]};
          mma_h(d, af, bf[q][2 * n2], bf[q][2 * n2 + 1]);
#pragma unroll
          for (int w = 0; w < 4; ++w) acc[n2][w][s + q] = d[w];
        }
    }
#pragma unroll
    for (int n2 = 0; n2 < 2; ++n2)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = rb + (lane >> 2) + 8 * h, cc = cb + 8 * n2 + 2 * (lane & 3);
        if (r >= nrows || cc >= ncols) continue;
        const int ea = xe[r];
        T c2[2];
        memcpy(c2, &c4[n2][h], sizeof c2);
        fold_entry(c2[0], acc[n2][2 * h], ea, ye[cc]);
        if (pair || cc + 1 < ncols) fold_entry(c2[1], acc[n2][2 * h + 1], ea, ye[cc + 1]);
        T* p = row(r) + cc;
        if (pair) {
          memcpy(&c4[n2][h], c2, sizeof c2);
          *(float4*)p = c4[n2][h];
        } else {
          p[0] = c2[0];
          if (cc + 1 < ncols) p[1] = c2[1];
        }
      }
  }
}

}  // namespace
}  // namespace nmc
