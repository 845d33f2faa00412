// The sweep's products with constant matrices, a whole matrix per CTA: wraps G <- B G B^{-1} (two
// products, constants left and right) and chains of block products X <- B_w ... B_1 U, for up to 112
// sites, in FP64 and in FP32 pairs. Between the products of one call nothing leaves the chip.
//
// The arithmetic is exact slicing (Ozaki et al., Numer. Algorithms 2012) on FP16 tensor-core operands:
// each row of the left operand and column of the right one, scaled by a power of two, is cut into
// balanced digits: for FP32 pairs 6 of 10 bits (|d| <= 512), for FP64 7 of 9 bits (|d| <= 256); what is
// left is below 2^-59 (2^-62) of the row's maximum. Digit products s + t < digits accumulate in FP32
// groups g = s + t by mma.sync: exact over 64 terms for g <= 3 with 9 bits (64 * 4 * 2^16 = 2^24), over
// 32 for g <= 1 with 10 (32 * 2 * 2^18; beyond, only if two thirds of all digits were largest at once);
// after so many terms multiples of 2^10 (2^9) are carried to the next group up (exact). The groups are
// joined as FP32 pairs, or in 64-bit integers. (9 bits for the pairs too, without carries: 3% faster,
// but the dropped group s + t = 6 is then 2^-51 of a result: errors of a wrap 3 times gemm_tc.cu's.)
//
// Layout: a matrix of up to 16 T sites is T warps of 16 rows each. The accumulators of a 16 x 16 tile
// are laid out over the lanes just as the left operand of the next product wants them, so a result is
// cut in registers and kept in shared memory as ready operand fragments (16 bytes per lane) that only its
// own warp reads; the constants' fragments are prepared once per context and read through L1. Only the
// matrix that comes from memory is staged digit by digit for ldmatrix.
//
// tcgen05 multiplies these tiles four times as fast but wants 128 rows and every digit through shared
// and tensor memory: gemm_tc.cu's form, one product per launch, spent 33 us on 512 matrices of 64
// sites against 5 us of tensor work, in its phases' latencies. It remains for more than 112 sites.
//
// us, product by product -> here: 512 matrices of 64 sites, a wrap 67 -> 47 (FP64 136 -> 68) and a chain
// of 10 332 -> 240 (FP64 680 -> 336); 1024 of 72 a wrap 300 -> 193, a chain of 10 1500 -> 1055; 128 of
// 100 91 -> 78, 455 -> 382; 2 of 16 in FP64 17 -> 8.4, 83 -> 22. The error of a wrap against long double,
// rms: pairs at 64 sites 3.6e-16 -> 2.1e-16 of the largest entry.
// What bounds it: the legacy tensor pipe (0.47 of its m16n8k16 instructions per cycle and SM), 23k of
// the 39k cycles that two matrices of 64 sites take on an SM together; staging, cutting and joining
// take the rest, side by side with the other CTA's products only by chance. 512 matrices are 1.7 rounds
// of 304 places, 72 sites leave a tenth of the tiles empty and five warps unevenly on four quarters.
#include <cuda_fp16.h>

#include <cstring>

#include "nmc_internal.cuh"
#include "wrap.cuh"

namespace nmc {

namespace {

NMC_DEBUG_FLAG

constexpr float kSplit = 12582912.f;   // 1.5 2^23: adding and removing it rounds to an integer

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

// (H 2^B + L) 2^k in FP64, rounded once, by integer operations (a conversion from 64 bits and a scaling
// would take the FP64 pipe) and without a branch, so that several sums interleave: outside FP64's normal
// range `slow` is set and join_slow gives the value.
template <int B>
__device__ __forceinline__ double join_fast(long long H, long long L, int k, bool& slow) {
  H += L >> B;
  L &= (1ll << B) - 1;
  const int s = min(__clzll(H ^ (H >> 63)) - 1, B);
  const long long v = (H << s) + (L >> (B - s));
  const unsigned long long m = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int z = __clzll(m), e = k + B - s - z + 1086;
  const unsigned long long t = m << (z & 63), f = (t >> 11) + ((t >> 10) & 1);
  const unsigned long long b = (((unsigned long long)(unsigned)(e - 1)) << 52) + f;
  slow |= v != 0 && (e < 1 || e > 2045);
  return __longlong_as_double(v == 0 ? 0ll : (long long)(b | ((unsigned long long)v & (1ull << 63))));
}
template <int B>
__device__ __noinline__ double join_slow(long long H, long long L, int k) {
  bool slow = false;
  const double fast = join_fast<B>(H, L, k, slow);
  if (!slow) return fast;
  H += L >> B;
  L &= (1ll << B) - 1;
  const int s = min(__clzll(H ^ (H >> 63)) - 1, B);
  return ldexp((double)((H << s) + (L >> (B - s))), k + B - s);
}

// What a value's digits are and how digit sums make a value
template <typename T> struct Cut;
template <> struct Cut<df2> {
  static constexpr int D = 6, W = 10, kCarry = 2, kMin = 9, kMax = 0xff;
  static __device__ __forceinline__ df2 zero() { return df2{0.f, 0.f}; }
  static __device__ __forceinline__ df2 mul(df2 a, df2 b) { return df_mul(a, b); }
  static __device__ __forceinline__ int expo(df2 a) { return (__float_as_int(a.hi) >> 23) & 0xff; }
  // digits in units of 2^(E - 135): rounding to multiples of 2^(-10 s) by a constant whose low mantissa
  // bits are 0x6600, FP16's 1536, leaves 1536 + digit in the low half. The low part joins by exact sums
  // (Fast2Sum: what is left of the high part is 0 or at least twice as large).
  static __device__ __forceinline__ void split(df2 a, float sc, unsigned (&t)[D]) {
    float v = __fmul_rn(a.hi, sc), e = __fmul_rn(a.lo, sc), m = __int_as_float(0x4b406600);
#pragma unroll
    for (int s = 0; s < D; ++s) {
      if (s >= 1 && s <= 3) {
        const float q = __fadd_rn(v, e);
        e = __fsub_rn(e, __fsub_rn(q, v));
        v = q;
      }
      if (s == 4) v = __fadd_rn(v, e);
      const float x = __fadd_rn(v, m);
      t[s] = __float_as_uint(x);
      v = __fsub_rn(v, __fsub_rn(x, m));
      m *= 0x1p-10f;
    }
  }
  static __device__ __forceinline__ void digits(df2 a, df2 b, int E, unsigned (&w)[D]) {
    const float sc = __int_as_float((262 - E) << 23);
    unsigned t0[D], t1[D];
    split(a, sc, t0);
    split(b, sc, t1);
#pragma unroll
    for (int s = 0; s < D; ++s) {
      const unsigned f = __byte_perm(t0[s], t1[s], 0x5410);
      const __half2 d = __hadd2(*reinterpret_cast<const __half2*>(&f), __float2half2_rn(-1536.f));
      w[s] = *reinterpret_cast<const unsigned*>(&d);
    }
  }
  // what the sums of a row (column) are multiplied by: 2^(E - 135), NaN where it holds a non-finite
  static __device__ __forceinline__ int scale(int E) { return E >= kMax ? 0x7fc00000 : (E - 8) << 23; }
  // sum_g a_g 2^(-10 g) times both scales; the first four groups by exact sums (Fast2Sum: where the
  // smaller operand comes first, the sum or its difference from that operand is short enough)
  static __device__ __forceinline__ df2 value(const float (&a)[D], int ea, int eb) {
    const float s = __fmaf_rn(a[1], 0x1p-10f, a[0]);
    const float e1 = __fmaf_rn(a[1], 0x1p-10f, -__fsub_rn(s, a[0]));
    const float h = __fmaf_rn(a[2], 0x1p-20f, s);
    const float e2 = __fmaf_rn(a[2], 0x1p-20f, -__fsub_rn(h, s));
    const float t = __fmaf_rn(a[3], 0x1p-30f, h);
    const float e3 = __fmaf_rn(a[3], 0x1p-30f, -__fsub_rn(t, h));
    float l = __fadd_rn(e1, __fadd_rn(e2, e3));
    l = __fadd_rn(l, __fmaf_rn(a[5], 0x1p-50f, __fmul_rn(a[4], 0x1p-40f)));
    const float sc = __fmul_rn(__int_as_float(ea), __int_as_float(eb));
    return df_norm(__fmul_rn(t, sc), __fmul_rn(l, sc));
  }
  // the same in FP64
  template <bool SLOW>
  static __device__ __forceinline__ double wide(const float (&a)[D], int ea, int eb, bool& slow) {
    int q[D];
#pragma unroll
    for (int s = 0; s < D; ++s) q[s] = __float2int_rn(a[s]);
    const long long H = (long long)q[0] * (1 << 20) + ((long long)q[1] * (1 << 10) + q[2]);
    const long long L = (long long)q[3] * (1 << 20) + ((long long)q[4] * (1 << 10) + q[5]);
    const int k = (ea >> 23) + (eb >> 23) - 254 - 50;
    const bool bad = ea == 0x7fc00000 || eb == 0x7fc00000;
    const double v = SLOW ? join_slow<30>(H, L, k) : join_fast<30>(H, L, k, slow);
    return bad ? __longlong_as_double(0x7ff8000000000000ll) : v;
  }
};
template <> struct Cut<double> {
  static constexpr int D = 7, W = 9, kCarry = 4, kMin = 1, kMax = 0x7ff;
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ int expo(double a) { return (__double2hiint(a) >> 20) & 0x7ff; }
  // digits in units of 2^(E - 1022 - 62): |x| plus 256 in every 9-bit field, the field less 256 with
  // x's sign (1024 + field is the FP16 whose mantissa is the field)
  static __device__ __forceinline__ void digits(double a, double b, int E, unsigned (&w)[D]) {
    unsigned long long u[2];
    unsigned short sg[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double x = q ? b : a;
      const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
      const int e = (int)((h >> 20) & 0x7ffu);
      const unsigned mh = __funnelshift_l(l, h, 11) | 0x80000000u;
      u[q] = (((unsigned long long)mh << 32 | (l << 11)) >> min(2 + E - e, 63)) + 0x4020100804020100ull;
      sg[q] = e == 0 ? 0 : (unsigned short)(0x3c00u | ((h >> 16) & 0x8000u));   // 0 or +-1
    }
    const __half2 sgn = __halves2half2(__ushort_as_half(sg[0]), __ushort_as_half(sg[1]));
    const __half2 off = __hmul2(sgn, __float2half2_rn(-1280.f));
#pragma unroll
    for (int s = 0; s < D; ++s) {
      const int bit = 9 * (D - 1 - s);
      unsigned f = __byte_perm((unsigned)(u[0] >> bit), (unsigned)(u[1] >> bit), 0x5410);
      if (s > 0) f &= 0x01ff01ffu;   // (the first digit's field may reach 512)
      f |= 0x64006400u;
      const __half2 d = __hfma2(*reinterpret_cast<__half2*>(&f), sgn, off);
      w[s] = *reinterpret_cast<const unsigned*>(&d);
    }
  }
  static __device__ __forceinline__ int scale(int E) { return E; }
  template <bool SLOW>
  static __device__ __forceinline__ double wide(const float (&a)[D], int ea, int eb, bool& slow) {
    int q[D];
#pragma unroll
    for (int s = 0; s < D; ++s) q[s] = __float2int_rn(a[s]);
    const long long H = (long long)q[0] * (1 << 18) + ((long long)q[1] * (1 << 9) + q[2]);
    const long long L = (long long)q[3] * (1 << 27) +
                        ((long long)q[4] * (1 << 18) + ((long long)q[5] * (1 << 9) + q[6]));
    // digit 0 counts units of 2^(E - 1022 - 8)
    const int k = ea + eb - 2 * 1030 - 54;
    const double v = SLOW ? join_slow<36>(H, L, k) : join_fast<36>(H, L, k, slow);
    return max(ea, eb) >= kMax ? __longlong_as_double(0x7ff8000000000000ll) : v;
  }
};

// Two warps share 16 rows for 4 tiles, one CTA's 8 warps on two of an SM's places: us, in pairs of warps / one
// warp to 16 rows, 512 matrices of 64 sites a wrap 48 / 61 (FP64 69 / 82) and a chain of ten 242 / 264 (334 /
// 350), 6 matrices 18 / 29 and 73 / 102. Elsewhere the tiles do not halve evenly or one warp has its rows alone
// and waits for no other: in an earlier form of these kernels pairs took 248 us against 183 for a wrap of 72
// sites x 1024, and 70 against 56 for chains of 36 x 128.
template <int T> constexpr int tiles_per_warp() { return T == 4 ? 2 : T; }

// A warp's tiles of a matrix of 16 T sites: 16 rows, H of the T columns of tiles
template <typename V, int T>
struct Tile {
  static constexpr int D = Cut<V>::D, Np = 16 * T, H = tiles_per_warp<T>(), NH = T / H;
  static constexpr int kThreads = 32 * T * NH;
  int N, mt, n0, lane;
  unsigned char* dig;   // digits: staged [digit][octet of k][vector][8], or fragments [mt][kt][digit][lane]
  int* ce;              // exponents of the staged vectors
  int* re;              // of the rows, two sets used in turn, where two warps share them
  int8_t* sg;           // signs of the slice's field times the spin

  __device__ __forceinline__ Tile(unsigned char* sm, int N_) : N(N_) {
    mt = (threadIdx.x >> 5) / NH;
    n0 = (threadIdx.x >> 5) % NH * H;
    lane = threadIdx.x & 31;
    dig = sm;
    ce = (int*)(sm + (size_t)D * Np * Np * 2);
    re = ce + Np;
    sg = (int8_t*)(re + 2 * Np);
    for (int i = threadIdx.x; i < 3 * Np; i += kThreads) ce[i] = Cut<V>::kMin;
  }
  // Stage X for ldmatrix: vectors n < N of N terms k. fetch(k, n) reads a term; after a barrier (what
  // `use` needs from the other threads is there), use(x, k, n) makes it the term staged.
  template <typename F, typename G>
  __device__ __forceinline__ void stage(F fetch, G use) {
    constexpr int kParts = kThreads / Np;                   // threads to a vector
    const int n = threadIdx.x % Np, q = threadIdx.x / Np;
    V x[H][8];
    int E = Cut<V>::kMin;
#pragma unroll
    for (int i = 0; i < H; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k = (q + kParts * i) * 8 + j;
        x[i][j] = n < N && k < N ? fetch(k, n) : Cut<V>::zero();
      }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < H; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int k = (q + kParts * i) * 8 + j;
        if (n < N && k < N) x[i][j] = use(x[i][j], k, n);
        E = max(E, Cut<V>::expo(x[i][j]));
      }
    atomicMax(&ce[n], E);
    __syncthreads();
    E = ce[n];
#pragma unroll
    for (int i = 0; i < H; ++i) {
      unsigned w[4][D];
#pragma unroll
      for (int p = 0; p < 4; ++p) Cut<V>::digits(x[i][2 * p], x[i][2 * p + 1], E, w[p]);
#pragma unroll
      for (int s = 0; s < D; ++s)
        *(uint4*)(dig + ((size_t)(s * 2 * T + q + kParts * i) * Np + n) * 16) =
            make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
    }
    __syncthreads();
  }
  // a staged 16 x 16 tile as left (rows v0 ..) or right (columns v0 ..) operand
  __device__ __forceinline__ void staged_left(unsigned (&f)[4], int v0, int kt, int s) const {
    ldm4(f, (unsigned)__cvta_generic_to_shared(dig) +
                ((s * 2 * T + 2 * kt + (lane >> 4)) * Np + v0 + (lane & 15)) * 16);
  }
  __device__ __forceinline__ void staged_right(unsigned (&f)[4], int v0, int kt, int s) const {
    ldm4(f, (unsigned)__cvta_generic_to_shared(dig) +
                ((s * 2 * T + 2 * kt + ((lane >> 3) & 1)) * Np + v0 + (lane & 7) + ((lane >> 4) & 1) * 8) * 16);
  }
  // a constant's tile (rows or columns 16 vt ..)
  __device__ __forceinline__ uint4 constant(const uint4* C, int vt, int kt, int s) const {
    return __ldg(C + ((vt * T + kt) * D + s) * 32 + lane);
  }
  // The warp's tiles y[tile][.], in the accumulators' layout, become the next left operand. set: which
  // set of row exponents, in turn (the other is reset).
  __device__ __forceinline__ void refragment(const V (&y)[H][8], int set, int& e0, int& e1) {
    int E[2] = {Cut<V>::kMin, Cut<V>::kMin};
#pragma unroll
    for (int j = 0; j < H; ++j)
#pragma unroll
      for (int e = 0; e < 8; ++e) E[(e >> 1) & 1] = max(E[(e >> 1) & 1], Cut<V>::expo(y[j][e]));
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      E[h] = max(E[h], __shfl_xor_sync(0xffffffffu, E[h], 1));
      E[h] = max(E[h], __shfl_xor_sync(0xffffffffu, E[h], 2));
    }
    if constexpr (NH > 1) {
      int* r = re + set * Np + mt * 16 + (lane >> 2);
      if ((lane & 3) == 0) {
        atomicMax(&r[0], E[0]);
        atomicMax(&r[8], E[1]);
      }
      rows_barrier();
      E[0] = r[0];
      E[1] = r[8];
      if (n0 == 0 && (lane & 3) == 0) {   // (read before the barrier that ends the previous call)
        int* o = re + (set ^ 1) * Np + mt * 16 + (lane >> 2);
        o[0] = o[8] = Cut<V>::kMin;
      }
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
      unsigned w[4][D];
#pragma unroll
      for (int p = 0; p < 4; ++p) Cut<V>::digits(y[j][2 * p], y[j][2 * p + 1], E[p & 1], w[p]);
#pragma unroll
      for (int s = 0; s < D; ++s)
        *(uint4*)(dig + ((size_t)((mt * T + n0 + j) * D + s) * 32 + lane) * 16) =
            make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
    }
    rows_barrier();
    e0 = Cut<V>::scale(E[0]);
    e1 = Cut<V>::scale(E[1]);
  }
  // of the warps that share these rows
  __device__ __forceinline__ void rows_barrier() const {
    if constexpr (NH == 1) __syncwarp();
    else asm volatile("bar.sync %0, %1;" ::"r"(1 + mt), "n"(32 * NH) : "memory");
  }
  __device__ __forceinline__ void fragment(unsigned (&f)[4], int kt, int s) const {
    const uint4 v = *(const uint4*)(dig + ((size_t)((mt * T + kt) * D + s) * 32 + lane) * 16);
    f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
  }
  // acc = the groups of tile nt of left x right
  template <typename FL, typename FR>
  __device__ __forceinline__ void groups(float (&acc)[2][4][D], int nt, FL left, FR right) const {
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
      for (int g = 0; g < D; ++g) acc[i >> 2][i & 3][g] = 0.f;
#pragma unroll 1
    for (int kt = 0; kt < T; ++kt) {
      if (T > Cut<V>::kCarry && kt > 0 && kt % Cut<V>::kCarry == 0) {   // carries
#pragma unroll
        for (int g = D - 1; g > 0; --g)
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float& a = acc[i >> 2][i & 3][g];
            const float c = __fsub_rn(__fmaf_rn(a, 1.f / (1 << Cut<V>::W), kSplit), kSplit);
            a = __fmaf_rn(c, -(float)(1 << Cut<V>::W), a);
            acc[i >> 2][i & 3][g - 1] += c;
          }
      }
      unsigned b[D][4];
#pragma unroll
      for (int s = 0; s < D; ++s) right(b[s], nt, kt, s);
#pragma unroll
      for (int s = 0; s < D; ++s) {
        unsigned a[4];
        left(a, kt, s);
#pragma unroll
        for (int q = 0; q + s < D; ++q)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float d[4] = {acc[h][0][s + q], acc[h][1][s + q], acc[h][2][s + q], acc[h][3][s + q]};
            mma_h(d, a, b[q][2 * h], b[q][2 * h + 1]);
#pragma unroll
            for (int w = 0; w < 4; ++w) acc[h][w][s + q] = d[w];
          }
      }
    }
  }
};

// A tile's 8 results on this lane, in FP64 (O = double) or as the matrices are held: ea0, ea1 the scales of
// its two rows, eb(e) those of the columns. All fast results first, so that they interleave.
template <typename V, typename O, typename F>
__device__ __forceinline__ void results(const float (&acc)[2][4][Cut<V>::D], int ea0, int ea1, F eb, O (&o)[8]) {
  bool slow = false;
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int ea = (e & 2) ? ea1 : ea0;
    if constexpr (std::is_same<O, double>::value) o[e] = Cut<V>::template wide<false>(acc[e >> 2][e & 3], ea, eb(e), slow);
    else o[e] = Cut<V>::value(acc[e >> 2][e & 3], ea, eb(e));
  }
  if constexpr (std::is_same<O, double>::value)
    if (slow) {
#pragma unroll
      for (int e = 0; e < 8; ++e)
        o[e] = Cut<V>::template wide<true>(acc[e >> 2][e & 3], (e & 2) ? ea1 : ea0, eb(e), slow);
    }
}

__host__ __device__ constexpr size_t tile_smem(int D, int Np) {
  return (size_t)D * Np * Np * 2 + 3 * Np * sizeof(int) + Np;
}

// CTAs to an SM, by registers and shared memory
template <int T> constexpr int min_ctas() { return T == 1 ? 12 : T == 2 ? 6 : T == 3 ? 4 : T == 4 ? 2 : T == 5 ? 2 : 1; }

template <typename V, int T>
__global__ void __launch_bounds__(Tile<V, T>::kThreads, min_ctas<T>())
k_wrap(const WrapArgs<V> g) {
  extern __shared__ __align__(16) unsigned char sm[];
  Tile<V, T> t(sm, g.N);
  const int N = g.N, b = blockIdx.x, lane = t.lane;
  const bool fl = g.fields != nullptr;
  if (fl) {
    const int8_t* f = g.fields + (long long)(g.ns == 2 ? b >> 1 : b) * g.fstride;
    const int spin = g.ns == 2 && (b & 1) ? -1 : 1;
    for (int i = threadIdx.x; i < N; i += Tile<V, T>::kThreads) t.sg[i] = (int8_t)(f[i] > 0 ? spin : -spin);
  }
  const V* X = g.X + (long long)b * g.sX;
  // e^{sigma lam (s_r - s_c)}: 1 or e^{+-2 lam}
  auto field = [&](V v, int r, int c) {
    return t.sg[r] == t.sg[c] ? v : Cut<V>::mul(v, t.sg[r] > 0 ? g.e2 : g.em2);
  };
  const bool before = fl && g.before;
  auto column = [&](int nt, int e) { return nt * 16 + (e >> 2) * 8 + 2 * (lane & 3) + (e & 1); };
  t.stage([&](int k, int n) { return X[k * N + n]; }, [&](V v, int k, int n) { return before ? field(v, k, n) : v; });

  constexpr int H = Tile<V, T>::H;
  V y[H][8];
  const int r0 = t.mt * 16 + (lane >> 2);
  {
    const int a0 = __ldg(g.Le + r0), a1 = __ldg(g.Le + r0 + 8);
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int nt = t.n0 + j;
      float acc[2][4][Cut<V>::D];
      t.groups(acc, nt,
               [&](unsigned (&f)[4], int kt, int s) {
                 const uint4 v = t.constant(g.L, t.mt, kt, s);
                 f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
               },
               [&](unsigned (&f)[4], int n, int kt, int s) { t.staged_right(f, n * 16, kt, s); });
      results<V>(acc, a0, a1, [&](int e) { return Cut<V>::scale(t.ce[column(nt, e)]); }, y[j]);
    }
  }
  __syncthreads();   // the staged digits are read: their place is the fragments'
  int e0, e1;
  t.refragment(y, 0, e0, e1);
#pragma unroll 1
  for (int nt = t.n0; nt < t.n0 + H; ++nt) {
    float acc[2][4][Cut<V>::D];
    t.groups(acc, nt, [&](unsigned (&f)[4], int kt, int s) { t.fragment(f, kt, s); },
             [&](unsigned (&f)[4], int n, int kt, int s) {
               const uint4 v = t.constant(g.R, n, kt, s);
               f[0] = v.x, f[1] = v.z, f[2] = v.y, f[3] = v.w;
             });
    auto eb = [&](int e) { return __ldg(g.Re + column(nt, e)); };
    // pairs of columns
    auto place = [&](int e, long long& idx) {
      const int r = r0 + (e & 2) * 4, c = column(nt, e);
      idx = (long long)b * N * N + (long long)r * N + c;
      return r < N && c < N && NMC_DCHECK(b < g.batch && c + 1 < N, 501);   // (N is even)
    };
    long long idx;
    if (g.Cd) {
      double o[8];
      results<V>(acc, e0, e1, eb, o);
#pragma unroll
      for (int e = 0; e < 8; e += 2)
        if (place(e, idx)) *(double2*)(g.Cd + idx) = make_double2(o[e], o[e + 1]);
    } else {
      V o[8];
      results<V>(acc, e0, e1, eb, o);
#pragma unroll
      for (int e = 0; e < 8; e += 2) {
        if (!place(e, idx)) continue;
        if (fl && !g.before) {   // e^{-V} C e^{V}
          o[e] = field(o[e], column(nt, e), r0 + (e & 2) * 4);
          o[e + 1] = field(o[e + 1], column(nt, e) + 1, r0 + (e & 2) * 4);
        }
        float4 v;
        memcpy(&v, &o[e], sizeof v);
        *(float4*)(g.C + idx) = v;
      }
    }
  }
}

__device__ __forceinline__ void from_double(double& y, double x) { y = x; }
__device__ __forceinline__ void from_double(df2& y, double x) { y = df_from_double(x); }

// Columns of X are the rows here: row m holds column m of X, its k-th term X[k][m]. After the staging
// a warp waits only for the one that shares its rows.
template <typename V, int T>
__global__ void __launch_bounds__(Tile<V, T>::kThreads, min_ctas<T>())
k_chain(const ChainArgs<V> g) {
  extern __shared__ __align__(16) unsigned char sm[];
  Tile<V, T> t(sm, g.N);
  const int N = g.N, b = blockIdx.x, lane = t.lane;
  const double* U = g.U + (long long)b * g.sU;
  const int8_t* f = g.fields + (long long)(g.ns == 2 ? b >> 1 : b) * g.fstride;
  const bool flip = g.ns == 2 && (b & 1);
  // e^{sigma lam s}
  auto field = [&](V v, int8_t s) { return Cut<V>::mul(v, (s > 0) != flip ? g.e1 : g.em1); };
  {
    const int8_t* s = f + (long long)g.l0 * N;
    t.stage([&](int k, int n) {
              V v;
              from_double(v, U[(long long)k * N + n]);
              return v;
            },
            [&](V v, int k, int n) { return g.before ? field(v, s[k]) : v; });
  }
  auto column = [&](int nt, int e) { return nt * 16 + (e >> 2) * 8 + 2 * (lane & 3) + (e & 1); };
  const int r0 = t.mt * 16 + (lane >> 2);
  int e0 = Cut<V>::scale(t.ce[r0]), e1 = Cut<V>::scale(t.ce[r0 + 8]);
  auto constant = [&](unsigned (&v4)[4], int n, int kt, int s) {
    const uint4 v = t.constant(g.L, n, kt, s);
    v4[0] = v.x, v4[1] = v.z, v4[2] = v.y, v4[3] = v.w;
  };
  constexpr int H = Tile<V, T>::H;
  for (int k = 0; k + 1 < g.w; ++k) {
    V y[H][8];
    const int8_t* s = f + (long long)(g.l0 + (g.before ? k + 1 : k) * g.dl) * N;
#pragma unroll
    for (int j = 0; j < H; ++j) {
      const int nt = t.n0 + j;
      float acc[2][4][Cut<V>::D];
      t.groups(acc, nt,
               [&](unsigned (&a)[4], int kt, int d) {
                 if (k == 0) t.staged_left(a, t.mt * 16, kt, d);
                 else t.fragment(a, kt, d);
               },
               constant);
      results<V>(acc, e0, e1, [&](int e) { return __ldg(g.Le + column(nt, e)); }, y[j]);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = column(nt, 4 * h);
        // one byte at a time: nmc_green_noalloc's caller may have the fields at any address (N is even)
        const int8_t s0 = c < N ? s[c] : 1, s1 = c < N ? s[c + 1] : 1;
#pragma unroll
        for (int i = 0; i < 4; ++i) y[j][4 * h + i] = field(y[j][4 * h + i], (i & 1) ? s1 : s0);
      }
    }
    if (k == 0) __syncthreads();   // the staged digits are read: their place is the fragments'
    t.refragment(y, k & 1, e0, e1);
  }
  // the last product, times D, in FP64
  const int8_t* s = f + (long long)(g.l0 + (g.w - 1) * g.dl) * N;
  const double d0 = r0 < N ? g.Dv[(long long)b * g.sD + r0] : 0.0;
  const double d1 = r0 + 8 < N ? g.Dv[(long long)b * g.sD + r0 + 8] : 0.0;
#pragma unroll 1
  for (int nt = t.n0; nt < t.n0 + H; ++nt) {
    float acc[2][4][Cut<V>::D];
    t.groups(acc, nt,
             [&](unsigned (&a)[4], int kt, int d) {
               if (g.w == 1) t.staged_left(a, t.mt * 16, kt, d);
               else t.fragment(a, kt, d);
             },
             constant);
    double o[8];
    results<V>(acc, e0, e1, [&](int e) { return __ldg(g.Le + column(nt, e)); }, o);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int c = column(nt, e), r = r0 + (e & 2) * 4;
      if (r >= N || c >= N || !NMC_DCHECK(b < g.batch, 502)) continue;
      double v = o[e] * ((e & 2) ? d1 : d0);
      if (!g.before) v *= (s[c] > 0) != flip ? g.d1 : g.dm1;
      g.X[(long long)b * N * N + (long long)c * N + r] = v;
    }
  }
}

// Fragments of a constant: vector v (row v of M, or column v with cols) and its terms k, zero beyond N
template <typename T>
__global__ void k_const_frags(const double* M, int N, int cols, uint4* out, int* scales) {
  constexpr int D = Cut<T>::D;
  const int T16 = (N + 15) >> 4, vt = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ int ev[16];
  auto at = [&](int v, int k) {
    T x = Cut<T>::zero();
    if (v < N && k < N) from_double(x, cols ? M[(long long)k * N + v] : M[(long long)v * N + k]);
    return x;
  };
  if (threadIdx.x < 16) {
    int E = Cut<T>::kMin;
    for (int k = 0; k < N; ++k) E = max(E, Cut<T>::expo(at(vt * 16 + threadIdx.x, k)));
    ev[threadIdx.x] = E;
    scales[vt * 16 + threadIdx.x] = Cut<T>::scale(E);
  }
  __syncthreads();
  for (int kt = warp; kt < T16; kt += blockDim.x >> 5) {
    unsigned w[4][D];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int v = (lane >> 2) + (p & 1) * 8, k = kt * 16 + (p >> 1) * 8 + 2 * (lane & 3);
      Cut<T>::digits(at(vt * 16 + v, k), at(vt * 16 + v, k + 1), ev[v], w[p]);
    }
#pragma unroll
    for (int s = 0; s < D; ++s)
      out[((vt * T16 + kt) * D + s) * 32 + lane] = make_uint4(w[0][s], w[1][s], w[2][s], w[3][s]);
  }
}

template <typename F> void by_tiles(int N, F run) {
  switch ((N + 15) / 16) {
    case 1: run(std::integral_constant<int, 1>()); break;
    case 2: run(std::integral_constant<int, 2>()); break;
    case 3: run(std::integral_constant<int, 3>()); break;
    case 4: run(std::integral_constant<int, 4>()); break;
    case 5: run(std::integral_constant<int, 5>()); break;
    case 6: run(std::integral_constant<int, 6>()); break;
    default: run(std::integral_constant<int, 7>()); break;
  }
}

}  // namespace

template <typename T> size_t frag_bytes(int N) {
  const size_t t = (N + 15) / 16;
  return t * t * Cut<T>::D * 32 * sizeof(uint4);
}
template size_t frag_bytes<double>(int);
template size_t frag_bytes<df2>(int);

template <typename T>
void prepare_frags(const double* M, int N, bool cols, void* frags, int* scales, cudaStream_t st) {
  k_const_frags<T><<<(N + 15) / 16, 128, 0, st>>>(M, N, cols, (uint4*)frags, scales);
}
template void prepare_frags<double>(const double*, int, bool, void*, int*, cudaStream_t);
template void prepare_frags<df2>(const double*, int, bool, void*, int*, cudaStream_t);

template <typename T>
void wrap_product(const WrapArgs<T>& g, cudaStream_t st) {
  by_tiles(g.N, [&](auto h) {
    constexpr int H = decltype(h)::value;   // tiles
    allow_max_dynamic_smem((const void*)k_wrap<T, H>);
    k_wrap<T, H><<<g.batch, Tile<T, H>::kThreads, tile_smem(Cut<T>::D, 16 * H), st>>>(g);
  });
}
template void wrap_product<double>(const WrapArgs<double>&, cudaStream_t);
template void wrap_product<df2>(const WrapArgs<df2>&, cudaStream_t);

template <typename T>
void chain_product(const ChainArgs<T>& g, cudaStream_t st) {
  by_tiles(g.N, [&](auto h) {
    constexpr int H = decltype(h)::value;   // tiles
    allow_max_dynamic_smem((const void*)k_chain<T, H>);
    k_chain<T, H><<<g.batch, Tile<T, H>::kThreads, tile_smem(Cut<T>::D, 16 * H), st>>>(g);
  });
}
template void chain_product<double>(const ChainArgs<double>&, cudaStream_t);
template void chain_product<df2>(const ChainArgs<df2>&, cudaStream_t);

NMC_DEBUG_READER(debug_fail_wrap)

}  // namespace nmc
