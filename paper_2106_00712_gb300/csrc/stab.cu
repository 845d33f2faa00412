// FP64 numerical stabilization of the DQMC sweep: UDV (here U D T) decompositions of the
// B-matrix products and the stable recompute of G = (I + R L)^{-1}.
//
// k_qrp: Householder QR with column pivoting (Businger-Golub): at step p the remaining
//   column of largest norm is swapped into place (norms are FP32, compared to 2^-19, lowest index on
//   ties: near-ties may fall either way, so D need not be ordered to the last bits), a reflector
//   H_p = I - tau v v^T zeroes it below the diagonal, and the trailing columns are updated;
//   squared column norms are downdated and summed again when little of them is left. Outputs
//   U = Q (column by column, in registers), D = |diag R| and
//   T = D^{-1} R P^T.
// k_solve: Y = X^{-1} (Db_R^{-1} U_R^T) by blocked LU with partial pivoting; X is the
//   well-scaled middle factor of the stabilized inverse, so partial pivoting is sufficient.
//
// One CTA per matrix (batch = 2 * chains); the working matrix lives in shared memory
// when it fits and in a per-matrix global workspace otherwise.
#include "fold16.cuh"
#include "nmc_internal.cuh"

#include <type_traits>

namespace nmc {

namespace {

NMC_DEBUG_FLAG

// Gauss-Jordan: 16 warps (rows over warps, columns over lanes), so a matrix alone on an SM
// (the tail of a batch that does not fill the GPU in one wave) still has the warps to hide
// the FP64 latency
constexpr int kSolveThreads = 512;
constexpr int kSolveWarps = kSolveThreads / 32;
constexpr size_t kSmemLimit = 200 * 1024;
// Up to here Gauss-Jordan is faster: 16 sites x 2 matrices 23 us against 29, 36 x 128 73 against 91;
// 48 x 6 110 against 111, 48 x 512 296 against 229.
constexpr int kGaussJordanMax = 40;
constexpr size_t kQrSmemLimit = 225 * 1024;

// ---------------------------------------------------------------------------- QR
// The FP64 pipe issues one warp operation per 20 cycles and SM, an integer multiply-add 32 x 32 +
// 64 bits one per 0.55, so the reflections run in fixed point: a column is held as 64-bit integers
// in units of 2^-58 of a power of two just above its 2-norm. Reflections preserve that norm, so
// nothing overflows, and every operation's error is at most a few 2^-58 of the column's norm,
// where an FP64 Householder QR makes a few 2^-53 of it. An integer is split into limbs
// c = c1 2^29 + c0 (|c1| <= 2^30, |c0| <= 2^28); a product takes three multiply-adds, c0 d0 being
// below the unit:  a b / 2^58 = a1 b1 + (a1 b0 + a0 b1) / 2^29.  The sums over a column cannot
// overflow: |sum a1 b1| <= |a| |b| / 2^58 (Cauchy-Schwarz), |sum a1 b0| <= 2^58 sqrt(N).
// A reflector is v = x - beta e_p shifted left until 2^58 <= |v| < 2^59 (exact), with
// tau = 2 / |v|^2 evaluated in integers from the entries actually stored.
//
// LPC lanes share a column (rows r = LPC j + lane, at most 4 NB each, held in registers between
// the dot product and the update), so a matrix of 64 columns keeps 256 threads busy; one warp
// searches the pivot and evaluates the reflector's scalars.
// What bounds it: one matrix, the serial chain of a step (pivot search, column norm, reflector, then
// the update, a barrier after each); many, the issue slots and the barriers around that chain.
// Measured, us per launch against an FP64 kernel with one thread per column (N, matrices): 361 / 722
// (64, 512), 1221 / 1904 (72, 1024), 560 / 1281 (100, 128), 42 / 71 (16, 2) and, with the matrix in
// global memory, where lanes along the rows read whole lines, 5034 / 87627 (256, 64). Those formed Q
// like R, one reflector on all columns and a barrier at a time; Q's columns are now each built in
// registers, the pivot column is read once, and what is in shared memory is so at compile time. On one
// set of graded and degenerate matrices, with the same bits: 45 -> 35 (16, 2), 143 -> 115 (36, 128),
// 291 -> 230 (64, 6), 414 -> 340 (64, 512), 422 -> 369 (72, 6), 1397 -> 1229 (72, 1024), 717 -> 619
// (100, 128), 1387 -> 1245 (144, 128), 5734 -> 5181 (256, 64), 37.5 -> 30.8 ms (512, 2); with the rows'
// loops without tests per block 33, 107, 195, 338, 275, 1137, 571, 1100, 3861 us and 23.5 ms.
// max |U^T U - I| 7e-17 against 8e-16, columns of U D T to 1.5e-16 against 9e-16 (N = 64).
constexpr int kLimb = 29, kFix = 58;

// c += a b, 32 x 32 + 64 bits
__device__ __forceinline__ void mad_wide(long long& c, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(c) : "r"(a), "r"(b));
}
__device__ __forceinline__ int2 limbs(long long c) {
  const int c1 = (int)((c + (1ll << (kLimb - 1))) >> kLimb);
  return make_int2(c1, (int)((unsigned)c - ((unsigned)c1 << kLimb)));
}
__device__ __forceinline__ long long fold(long long hi, long long mid) {
  return hi + ((mid + (1ll << (kLimb - 1))) >> kLimb);
}
// x in units of 2^(Eb - 1022 - 58) (|x| < 2^(Eb - 1022)), to nearest
__device__ __forceinline__ long long to_fixed(double x, int Eb) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const int e = (int)((h >> 20) & 0x7ffu);
  const unsigned mh = __funnelshift_l(l, h, 11) | 0x80000000u;
  const int sh = min(63 - kFix + Eb - e, 63);   // to 59 bits, then rounded to 58
  const unsigned long long m = ((((unsigned long long)mh << 32) | (l << 11)) >> sh) + 1ull;
  const long long v = e == 0 ? 0 : (long long)(m >> 1);
  return (int)h < 0 ? -v : v;
}
// v 2^k, with a result outside the normal range left to ldexp
__device__ __forceinline__ double pow2_scale(double v, int k) {
  const int e = (__double2hiint(v) >> 20) & 0x7ff;
  if (((__double2hiint(v) << 1) | __double2loint(v)) == 0) return v;
  if (e == 0 || e == 0x7ff || e + k < 1 || e + k > 2046) return ldexp(v, k);
  return __hiloint2double(__double2hiint(v) + k * (1 << 20), __double2loint(v));
}
// key of a squared norm n 4^E (n >= 0 a float): orders like the value to 2^-19, 0 for 0
__device__ __forceinline__ unsigned norm_key(float n, int Eb) {
  return n > 0.f ? (__float_as_uint(n) >> 4) + ((unsigned)(2 * Eb) << 19) : 0u;
}
// sum of a 64-bit integer over the warp, in every lane, by 32-bit warp reductions of 26-bit parts
__device__ __forceinline__ long long warp_sum64(long long v) {
  const unsigned m = (1u << 26) - 1;
  const unsigned a = __reduce_add_sync(0xffffffffu, (unsigned)v & m);
  const unsigned b = __reduce_add_sync(0xffffffffu, (unsigned)(v >> 26) & m);
  const int c = __reduce_add_sync(0xffffffffu, (int)(v >> 52));
  return (long long)a + ((long long)b << 26) + ((long long)c << 52);
}
// c + a b / 2^58 for a given by its limbs and b by its limbs
__device__ __forceinline__ long long madq(long long c, int2 a, int2 b) {
  long long mid = 1ll << (kLimb - 1);
  mad_wide(c, a.x, b.x);
  mad_wide(mid, a.x, b.y);
  mad_wide(mid, a.y, b.x);
  return c + (mid >> kLimb);
}
typedef unsigned long long u64;
typedef unsigned __int128 u128;
__device__ __forceinline__ int clz128(u128 v) {
  const u64 h = (u64)(v >> 64);
  return h ? __clzll((long long)h) : 64 + __clzll((long long)(u64)v);
}
__device__ __forceinline__ u128 shift128(u128 v, int right) {
  return right >= 0 ? v >> right : v << -right;
}
// sqrt(S), rounded, and 2^121 / n for n in [2^62, 2^64), by one third-order Newton step in 64-bit
// integers from an FP32 approximation (relative error e < 2^-20, so e^3 is below the last bit).
// The FP64 unit's latency (about 70 cycles an operation) would make these two the longest part
// of a reflection.
__device__ __forceinline__ u64 isqrt128(u128 S) {
  const int sh = (64 - clz128(S) + 1) & ~1;          // even: m = S 2^-sh in [2^62, 2^64)
  const u64 m = (u64)shift128(S, sh);
  const u64 Y = (u64)__float2uint_rn(rsqrtf((float)(unsigned)(m >> 32)) * 0x1p39f);
  const long long e = (1ll << 61) - (long long)__umul64hi(m, (Y * Y) << 15);   // 2^61 (1 - m y^2)
  const int es = (int)(e >> 10);
  const long long c = (e >> 1) + ((3 * (((long long)es * es) >> 41)) >> 3);
  const u64 y = (Y << 38) + (u64)(((long long)Y * (c >> 1)) >> 22);            // 1/sqrt, 2^77 units
  const u64 r = __umul64hi(m, y << 1);                                         // sqrt(m) 2^30
  const int d = 30 - sh / 2;
  return (r + ((1ull << d) >> 1)) >> d;
}
__device__ __forceinline__ long long recip121(u64 n) {
  const u64 Z = (u64)__float2uint_rn(__frcp_rn((float)(unsigned)(n >> 32)) * 0x1p55f);
  const long long e = (1ll << 61) - (long long)__umul64hi(n, Z << 38);         // 2^61 (1 - n z)
  const int es = (int)(e >> 10);
  const long long c = e + (((long long)es * es) >> 41);
  return (long long)(Z << 34) + (((long long)Z * (c >> 3)) >> 24);
}

// column stride: all rows a lane may touch (the padding is zero), the columns of a half warp on
// different banks
__host__ __device__ constexpr int qr_ld(int rows, int LPC) { return LPC < 16 ? rows + LPC : rows; }
__host__ __device__ constexpr size_t qr_small_bytes(int rows, int N) {
  // reflector (two buffers), its head and tau per column, norms, exponents, permutation
  return (size_t)rows * 2 * 8 + (size_t)N * (2 * 8 + 2 * 4 + 2 * 4);
}

// The working matrix is in shared memory up to 160 sites (8 lanes), which is all that fits.
__host__ __device__ constexpr bool qr_smem(int LPC) { return LPC < 16; }
static_assert(((qr_small_bytes(160, 160) + 15) & ~(size_t)15) + 160 * qr_ld(160, 8) * 8 <= kQrSmemLimit, "");

// f(block number as a type) for the first block bs in [B, NB): one straight run of code for each first
// block, where a test per block would keep a block's loads from starting before the last one's sums
template <int B, int NB, class F>
__device__ __forceinline__ void from_block(int bs, F&& f) {
  if constexpr (B + 1 < NB) {
    if (bs > B) {
      from_block<B + 1, NB>(bs, f);
      return;
    }
  }
  f(std::integral_constant<int, B>{});
}

// dot product of a column, x in registers, and a reflector's limbs, as hi + mid / 2^29, in this lane's
// rows of the blocks from B on
template <int B, int NB, int LPC>
__device__ __forceinline__ void dot_rows(const long long (&x)[NB][4], const int2* v, long long& hi, long long& mid) {
  long long m0 = 0, m1 = 0;   // two chains (wrapping sums: any order gives the same)
  hi = 0;
#pragma unroll
  for (int q = B; q < NB; ++q)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int2 l = limbs(x[q][i]), w = v[(4 * q + i) * LPC];
      mad_wide(hi, w.x, l.x);
      mad_wide(m0, w.x, l.y);
      mad_wide(m1, w.y, l.x);
    }
  mid = m0 + m1;
#pragma unroll
  for (int o = 1; o < LPC; o <<= 1) {
    hi += __shfl_xor_sync(0xffffffffu, hi, o);
    mid += __shfl_xor_sync(0xffffffffu, mid, o);
  }
}

template <int LPC, int NB, int THREADS, int CTAS>
__global__ void __launch_bounds__(THREADS, CTAS)
k_qrp(const double* __restrict__ X, double* __restrict__ U, double* __restrict__ D,
      double* __restrict__ Tp, double* __restrict__ ws, int N) {
  constexpr int kRows = 4 * NB * LPC, ldw = qr_ld(kRows, LPC), ngrp = THREADS / LPC;
  constexpr int kPer = (kRows + 31) / 32;        // rows per lane when a warp holds a column
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int2 s_tau;
  __shared__ int s_bad;
  const int b = blockIdx.x;
  const long long NN = (long long)N * N;
  int2* vl = (int2*)smraw;                       // [2][kRows] limbs of a reflector, zero elsewhere
  int2* vhead = vl + 2 * kRows;                  // [N] v_p
  int2* taus = vhead + N;                        // [N]
  float* n1 = (float*)(taus + N);                // [N] squared norms of the trailing part, of 4^E
  float* n2 = n1 + N;                            // [N] the same when last summed
  int* Eb = (int*)(n2 + N);                      // [N] biased exponent of the column's scale
  int* perm = Eb + N;                            // [N]
  long long* W;
  if constexpr (qr_smem(LPC)) W = (long long*)(smraw + ((qr_small_bytes(kRows, N) + 15) & ~(size_t)15));
  else W = (long long*)(ws + (long long)b * 2 * NN);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int sub = tid % LPC, grp = tid / LPC, wgrp = warp * 32 / LPC;   // the warp's first group
  // the serial warp: on another sub-partition in each of the CTAs that share an SM (warp w issues
  // on w % 4)
  const int pw = blockIdx.x & 3 & (THREADS / 32 - 1);
  const double* Xb = X + (long long)b * NN;

  if (tid == 0) s_bad = 0;
  for (int e = tid; e < (int)NN; e += THREADS) {
    const int r = e / N, c = e - r * N;
    ((double*)W)[(long long)c * ldw + r] = Xb[e];
  }
  for (int e = tid; e < N * (kRows - N); e += THREADS)
    W[(long long)(e / (kRows - N)) * ldw + N + e % (kRows - N)] = 0;
  for (int r = tid; r < 2 * kRows; r += THREADS) vl[r] = make_int2(0, 0);
  for (int c = tid; c < N; c += THREADS) perm[c] = c;
  __syncthreads();
  // columns to fixed point: the scale from the largest entry, raised to the 2-norm
  for (int c0 = 0; c0 < N; c0 += ngrp) {
    const int c = c0 + grp;
    long long* col = W + (long long)min(c, N - 1) * ldw;
    int em = 1;
    for (int r = sub; r < N; r += LPC) em = max(em, (int)(((unsigned)((int2*)col)[r].y >> 20) & 0x7ffu));
#pragma unroll
    for (int o = 1; o < LPC; o <<= 1) em = max(em, __shfl_xor_sync(0xffffffffu, em, o));
    float s = 0.f;   // of 4^em
    for (int r = sub; r < N; r += LPC) {
      const float y = (float)(int)(to_fixed(((double*)col)[r], em) >> 28) * 0x1p-30f;
      s = fmaf(y, y, s);
    }
#pragma unroll
    for (int o = 1; o < LPC; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    int up = 0;
    float sn = s * 1.00001f;
    while (sn > 1.f) sn *= 0.25f, s *= 0.25f, ++up;
    if (c < N) {
      for (int r = sub; r < N; r += LPC) col[r] = to_fixed(((double*)col)[r], em + up);
      if (sub == 0) {
        Eb[c] = em + up;
        n1[c] = n2[c] = s;
        if (em == 0x7ff) s_bad = 1;   // an infinity or a NaN: the outputs are NaN
      }
    }
  }
  __syncthreads();

  for (int p = 0; p < N; ++p) {
    int2* vp = vl + (p & 1) * kRows;
    if (warp == pw) {
      // pivot (largest trailing norm, lowest index on ties) and swap
      unsigned best = 0;
      int bi = p;
      for (int c = p + lane; c < N; c += 32) {
        const unsigned kc = norm_key(n1[c], Eb[c]);
        if (kc > best) { best = kc; bi = c; }
      }
      const unsigned top = __reduce_max_sync(0xffffffffu, best);
      bi = top == 0 ? p : (int)__reduce_min_sync(0xffffffffu, best == top ? (unsigned)bi : 0xffffu);
      const int piv = NMC_DCHECK(bi >= p && bi < N, 201) ? bi : p;
      long long* col = W + (long long)p * ldw;
      long long* other = W + (long long)piv * ldw;
      const long long alpha = other[p];
      long long y[kPer];   // the pivot column; column p takes its place
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int r = lane + 32 * i;
        y[i] = r < N ? other[r] : 0;
      }
      __syncwarp();
      if (piv != p) {
#pragma unroll
        for (int i = 0; i < kPer; ++i) {
          const int r = lane + 32 * i;
          if (r < N) {
            other[r] = col[r];
            if (r < p) col[r] = y[i];
          }
        }
        if (lane == 0) {
          n1[piv] = n1[p];
          n2[piv] = n2[p];
          int t = Eb[p]; Eb[p] = Eb[piv]; Eb[piv] = t;
          t = perm[p]; perm[p] = perm[piv]; perm[piv] = t;
        }
      }
      // squared norm from the diagonal down, exactly: HI 2^58 + MID 2^30 + LO
      long long hi = 0, mid = 0, lo = 0;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int2 c = limbs(lane + 32 * i >= p ? y[i] : 0);
        mad_wide(hi, c.x, c.x);
        mad_wide(mid, c.x, c.y);
        mad_wide(lo, c.y, c.y);
      }
      mid += lo >> 30;   // (LO's sum over the warp stays in range)
      lo &= (1ll << 30) - 1;
      hi = warp_sum64(hi);
      mid = warp_sum64(mid);
      lo = warp_sum64(lo);
      int k = 0;
      long long head = 0, beta = 0;
      int2 tau = make_int2(0, 0);
      if ((hi | mid | lo) != 0) {
        const u128 S = ((u128)hi << 58) + (u128)((__int128)mid << 30) + (u128)lo;
        const u64 root = isqrt128(S), al = (u64)(alpha < 0 ? -alpha : alpha);
        beta = alpha > 0 ? -(long long)root : (long long)root;
        head = alpha - beta;   // no cancellation
        // |v|^2 before the shift, exactly: S + 2 |alpha| |beta| + beta^2, with beta as stored
        const u128 V = S + (u128)root * (root + 2 * al);
        k = (clz128(V) - 10) >> 1;           // 2^116 <= V 4^k < 2^118
        tau = limbs(recip121((u64)shift128(V, 54 - 2 * k)));
        head = k >= 0 ? head << k : head >> -k;
      }
      __syncwarp();
      // the reflector's limbs, for this step and (below the diagonal) for Q
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        const int r = lane + 32 * i;
        if (r > p && r < N) {
          const int2 l = limbs(k >= 0 ? y[i] << k : y[i] >> -k);
          vp[r] = l;
          ((int2*)col)[r] = l;
        }
      }
      if (lane == 0) {
        const int2 hl = limbs(head);
        col[p] = beta;
        vp[p] = hl;
        vhead[p] = hl;
        taus[p] = tau;
        s_tau = tau;
        if (p >= 2) vp[p - 2] = make_int2(0, 0);   // what this buffer last held above row p
        if (p >= 1) vp[p - 1] = make_int2(0, 0);
      }
    }
    __syncthreads();
    const int2 tau = s_tau;
    const int bs = p / (4 * LPC);   // blocks of 4 LPC rows from here on
    for (int c0 = p + 1; c0 + wgrp < N; c0 += ngrp) {
      const int c = min(c0 + grp, N - 1);
      const bool on = c0 + grp < N;
      long long* col = W + (long long)c * ldw + sub;
      const int2* v = vp + sub;
      const float a2 = n2[c], a0 = n1[c];
      from_block<0, NB>(bs, [&](auto first) {
        constexpr int B = decltype(first)::value;
        long long x[NB][4], hi, mid;
#pragma unroll
        for (int q = B; q < NB; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i) x[q][i] = col[(4 * q + i) * LPC];
        dot_rows<B, NB, LPC>(x, v, hi, mid);
        const int2 f = limbs(-madq(0, limbs(fold(hi, mid)), tau));
#pragma unroll
        for (int q = B; q < NB; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i) {   // (rows above p: v is zero there)
            x[q][i] = madq(x[q][i], v[(4 * q + i) * LPC], f);
            if (on) col[(4 * q + i) * LPC] = x[q][i];
          }
        // trailing norm: downdated by row p's entry, summed again when less than 2^-12 of the last
        // sum is left
        __syncwarp();
        const float rp = (float)(col - sub)[p] * 0x1p-58f;
        float a1 = fmaf(-rp, rp, a0);
        const bool again = on && !(a1 > 0x1p-12f * a2);
        if (__any_sync(0xffffffffu, again)) {
          float s = 0.f;
#pragma unroll
          for (int q = B; q < NB; ++q)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float y = (4 * q + i) * LPC + sub > p ? (float)x[q][i] * 0x1p-58f : 0.f;
              s = fmaf(y, y, s);
            }
#pragma unroll
          for (int o = 1; o < LPC; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
          if (again && sub == 0) n2[c] = s;
          if (again) a1 = s;
        }
        if (on && sub == 0) n1[c] = a1;
      });
    }
    __syncthreads();
  }

  // outputs D = |diag R| and T = D^{-1} R P^T
  const bool bad = s_bad != 0;
  const double nan = __longlong_as_double(0x7ff8000000000000ll);
  double* Db = D + (long long)b * N;
  double* Tb = Tp + (long long)b * NN;
  double2* rd = (double2*)vl;   // |R_rr| and its reciprocal
  for (int r = tid; r < N; r += THREADS) {
    const double d = fabs((double)W[(long long)r * ldw + r]);
    Db[r] = bad ? nan : pow2_scale(d, Eb[r] - 1022 - kFix);
    rd[r] = make_double2(d, 1.0 / d);
  }
  __syncthreads();
  for (int e = tid; e < (int)NN; e += THREADS) {
    const int r = e / N, c = e - r * N;
    double t = 0.0;
    if (c >= r) {   // the quotient from the reciprocal, corrected by its remainder (as in quotient.cuh)
      const double w = (double)W[(long long)c * ldw + r], d = rd[r].x;
      t = w * rd[r].y;
      t = pow2_scale(fma(fma(-t, d, w), rd[r].y, t), Eb[c] - Eb[r]);
    }
    Tb[r * N + perm[c]] = bad ? nan : t;
  }
  __syncthreads();   // T and D are out: W's upper triangle is free
  // Q = H_0 H_1 ... H_{N-1}, 1 = 2^58: column c is H_0 ... H_c e_c (the later ones leave e_c alone),
  // so columns need nothing from each other: LPC lanes hold one in registers from e_c on, without a
  // barrier, the warp's 32 / LPC columns starting together (a reflection that comes too early for a
  // column multiplies zeros). With one column per group the second four of every eight warps take
  // their blocks backwards, so that each quarter of the SM (warp w on w % 4) gets long and short
  // ones; with several, rounds alternate. Against applying each reflector to all columns, a barrier
  // apiece: see the figures above.
  for (int c = warp; c < N; c += THREADS / 32) {   // whole reflectors, zero above the diagonal
    int2* v = (int2*)(W + (long long)c * ldw);
    for (int r = lane; r < c; r += 32) v[r] = make_int2(0, 0);
    if (lane == 0) v[c] = vhead[c];
  }
  __syncthreads();
  constexpr int nw = THREADS / 32, wcols = 32 / LPC;
  double* Ub = U + (long long)b * NN;
  for (int rd = 0; rd * ngrp < N; ++rd) {
    const int slot = N <= ngrp ? (warp & 4 ? min(warp | 3, nw - 1) - (warp & 3) : warp)
                               : (rd & 1 ? nw - 1 - warp : warp);
    const int cw = (rd * nw + slot) * wcols, c = cw + lane / LPC;
    if (cw >= N) continue;
    long long x[NB][4];
#pragma unroll
    for (int q = 0; q < NB; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) x[q][i] = (4 * q + i) * LPC + sub == c ? 1ll << kFix : 0;
    for (int p = min(cw + wcols, N) - 1; p >= 0; --p) {
      const int2 tau = taus[p];
      const int2* v = (const int2*)(W + (long long)p * ldw) + sub;
      from_block<0, NB>(p / (4 * LPC), [&](auto first) {
        constexpr int B = decltype(first)::value;
        long long hi, mid;
        dot_rows<B, NB, LPC>(x, v, hi, mid);
        const int2 f = limbs(-madq(0, limbs(fold(hi, mid)), tau));
#pragma unroll
        for (int q = B; q < NB; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i) x[q][i] = madq(x[q][i], v[(4 * q + i) * LPC], f);
      });
    }
    if (c < N) {
#pragma unroll
      for (int q = 0; q < NB; ++q)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = (4 * q + i) * LPC + sub;
          if (r < N) Ub[(long long)r * N + c] = bad ? nan : pow2_scale((double)x[q][i], -kFix);
        }
    }
  }
}

// argmax over lanes: larger key wins, lower index on ties. Keys are the bit patterns of
// non-negative doubles (|x|, squared norms), which order like the values, so the search
// runs on the integer pipes instead of the narrow FP64 pipe; a lane with no candidate
// holds key -1.
__device__ __forceinline__ void warp_argmax(long long& key, int& idx) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const long long ok = __shfl_xor_sync(0xffffffffu, key, o);
    const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
    if (ok > key || (ok == key && oi < idx)) { key = ok; idx = oi; }
  }
}

// key of a non-negative double (a NaN, with its sign bit cleared, orders above +inf)
__device__ __forceinline__ long long nonneg_key(double x) {
  return __double_as_longlong(x) & 0x7fffffffffffffffll;
}

// Few sites: Gauss-Jordan elimination with partial pivoting, one column at a time.
__global__ void __launch_bounds__(kSolveThreads)
k_solve_gj(const double* __restrict__ X, const double* __restrict__ UR, long long sUR,
           const double* __restrict__ DR, long long sDR, double* __restrict__ Y, int N) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_piv;
  __shared__ double s_inv;
  const int b = blockIdx.x;
  const long long NN = (long long)N * N;
  const int ld = 2 * N;
  double* Aug = (double*)smraw;  // row-major N x 2N
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const double* Xb = X + (long long)b * NN;
  const double* Ub = UR + (long long)b * sUR;
  const double* Dv = DR + (long long)b * sDR;
  for (int e = tid; e < 2 * (int)NN; e += kSolveThreads) {
    const int r = e / ld, c = e - r * ld;
    double v;
    if (c < N) v = Xb[r * N + c];
    else v = Ub[(c - N) * N + r] / fmax(Dv[r], 1.0);  // (Db_R^{-1} U_R^T)[r][c-N]
    Aug[e] = v;
  }
  __syncthreads();
  const int pw = blockIdx.x & 3;   // the pivot-search warp (see k_qrp)
  for (int p = 0; p < N; ++p) {
    if (warp == pw) {
      long long best = -1;
      int bi = p;
      for (int r = p + lane; r < N; r += 32) {
        const long long kr = nonneg_key(Aug[(long long)r * ld + p]);   // |entry|
        if (kr > best) { best = kr; bi = r; }
      }
      warp_argmax(best, bi);
      // the pivot's reciprocal, once: a division on every warp would cost the narrow FP64
      // pipe about as much as the elimination step itself
      if (lane == 0) {
        if (!NMC_DCHECK(bi >= p && bi < N, 202)) bi = p;
        s_piv = bi;
        s_inv = 1.0 / Aug[(long long)bi * ld + p];
      }
    }
    __syncthreads();
    const int piv = s_piv;
    if (piv != p) {
      for (int c = p + tid; c < ld; c += kSolveThreads) {
        const double t = Aug[(long long)p * ld + c];
        Aug[(long long)p * ld + c] = Aug[(long long)piv * ld + c];
        Aug[(long long)piv * ld + c] = t;
      }
      __syncthreads();
    }
    const double inv = s_inv;
    for (int c = p + 1 + tid; c < ld; c += kSolveThreads) Aug[p * ld + c] *= inv;
    __syncthreads();
    // rows over warps, columns over lanes (32-bit indices)
    for (int r = warp; r < N; r += kSolveWarps) {
      if (r == p) continue;
      const double mlt = Aug[r * ld + p];
      for (int c = p + 1 + lane; c < ld; c += 32) Aug[r * ld + c] -= mlt * Aug[p * ld + c];
    }
    __syncthreads();
  }
  double* Yb = Y + (long long)b * NN;
  for (int e = tid; e < (int)NN; e += kSolveThreads) {
    const int r = e / N, c = e - r * N;
    Yb[e] = Aug[r * ld + N + c];
  }
}

// ---------------------------------------------------------------------------- solve
// Y = X^{-1} (Db_R^{-1} U_R^T) by blocked LU with partial pivoting on the augmented matrix [X | RHS],
// 16 columns per block:
//   panel     thread t holds row t's 16 entries in registers; per column the pivot is the row with the
//             largest |entry| (its upper 32 bits; lowest index on ties), found per warp and then over
//             the warps' candidates, which bring their rows and reciprocals along: one barrier a column;
//             rows stay where they are, `map` says which one is k-th
//   rows      a thread per column solves the block's unit lower triangle (FP64) for its 16 rows
//   update    rows below -= (rows x 16) (16 x columns): fold16.cuh's tensor-core rank-16 update, the
//             digits cut from the registers of the two steps before
// then the triangular solve upwards over the blocks, with the same update of the rows above.
//
// Elimination in FP64 throughout took 1.5 N^3 multiply-adds at one warp operation per 20 cycles and
// SM (246k cycles a matrix at N = 64); here the FP64 pipe adds once per entry and block (28k), and
// does the triangles (48k) and the panels (26k).
// us, Gauss-Jordan -> here: 64 sites x 512 583 -> 335, 64 x 6 197 -> 155, 72 x 1024 1430 -> 971,
// 100 x 128 582 -> 313, 144 x 128 2800 -> 619, 256 x 64 (in global memory) 16100 -> 2150; the error of
// Y against 64-bit-mantissa elimination is about half of before. (With the pivots' reciprocals from an
// approximation, an ulp off and wrong for the smallest and largest, 325, 151, 926, 305, 606, 2121.)
// What bounds it: a matrix's dependent chain. Of 310k cycles at N = 64 the panels take 105k (1600 a
// column: search, division, barrier, and some ten FP64 operations at 80 cycles from one warp), the
// triangles 80k, the updates 70k; two matrices on an SM run in the time of one.
__host__ __device__ inline size_t solve_small_bytes(int N, int chunk, int nw) {
  const int rows = max((N - 1) & ~15, 16);   // digit rows: all but the first (last) block's
  return (size_t)kFDig * 32 * (rows + chunk) + 4 * (rows + chunk)       // digits, scales
         + 16 * 16 * 8 + 2 * nw * (16 * 8 + 16)                         // triangle, candidates
         + (size_t)N * 8 + (size_t)((N + 3) & ~3) * 4 + 64;             // 1 / pivots, row map, block's pivots
}

// RP: rows per thread of a panel. lda: row stride of the augmented matrix; chunk: columns whose digits
// are held at a time (a multiple of 16).
template <int THREADS, int RP, int CTAS, bool SMEM>
__global__ void __launch_bounds__(THREADS, CTAS)
k_solve(const double* __restrict__ X, const double* __restrict__ UR, long long sUR,
        const double* __restrict__ DR, long long sDR, double* __restrict__ Y,
        double* __restrict__ ws, int N, int lda, int chunk) {
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NW = THREADS / 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const long long NN = (long long)N * N;
  const int rows = max((N - 1) & ~15, 16), rs = rows * 32, cs = chunk * 32;
  double* A;   // row-major N x 2N
  if constexpr (SMEM) A = (double*)smraw;
  else A = ws + (long long)b * 2 * NN;
  unsigned char* rd = smraw + (SMEM ? (size_t)N * lda * sizeof(double) : 0);   // digits of rows
  unsigned char* cd = rd + (size_t)kFDig * rs;                                 // and of columns
  double (*tri)[16] = (double (*)[16])(cd + (size_t)kFDig * cs);   // the block's L (unit) below U
  double (*cand)[NW][16] = (double (*)[NW][16])(tri + 16);         // [parity][warp]: candidate's row
  double (*cinv)[NW] = (double (*)[NW])(cand + 2);                 // its entry's reciprocal
  unsigned (*ckey)[NW] = (unsigned (*)[NW])(cinv + 2);             // its key
  int (*cwho)[NW] = (int (*)[NW])(ckey + 2);                       // its row, counted from the block's first
  double* inv = (double*)(cwho + 2);                               // 1 / U_kk
  int* re = (int*)(inv + N);                                       // scales of digit rows, columns
  int* ce = re + rows;
  int* map = ce + chunk;                                           // storage row of the k-th row
  int* who = map + ((N + 3) & ~3);                                 // the block's pivots
  const unsigned rda = (unsigned)__cvta_generic_to_shared(rd), cda = (unsigned)__cvta_generic_to_shared(cd);

  const double* Xb = X + (long long)b * NN;
  const double* Ub = UR + (long long)b * sUR;
  const double* Dv = DR + (long long)b * sDR;
  for (int r = tid; r < N; r += THREADS) {
    map[r] = r;
    inv[r] = 1.0 / fmax(Dv[r], 1.0);
  }
  __syncthreads();
  for (int r = warp; r < N; r += NW)
    for (int c = lane; c < N; c += 32) {
      A[(long long)r * lda + c] = Xb[(long long)r * N + c];
      A[(long long)c * lda + N + r] = Ub[(long long)r * N + c] * inv[c];   // (Db_R^{-1} U_R^T)[c][r]
    }
  __syncthreads();

  // digits of w columns from column j0 on, of the 16 rows k0 ..
  auto cut_columns = [&](int j0, int w, int k0) {
    for (int c = tid; c < w; c += THREADS) {
      double x[16];
      int E = Digits<double>::kExpMin;
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        x[q] = k0 + q < N ? A[(long long)map[k0 + q] * lda + j0 + c] : 0.0;
        E = max(E, Digits<double>::expo(x[q]));
      }
      ce[c] = Digits<double>::scale(E);
      cut16<double>(x, E, cd, c, cs);
    }
  };

  for (int k0 = 0; k0 < N; k0 += 16) {
    const int kw = min(16, N - k0), left = N - k0;
    // ------------------------------------------------------------ panel
    double a[RP][16];
    int place[RP];   // -1: still a candidate; otherwise its place among the block's pivots
    int row[RP];
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int t = tid + i * THREADS;
      place[i] = t < left ? -1 : 16;
      row[i] = t < left ? map[k0 + t] : 0;
      const double* src = A + (long long)row[i] * lda + k0;
#pragma unroll
      for (int c = 0; c < 16; ++c) a[i][c] = t < left && c < kw ? src[c] : 0.0;
    }
    const int nw = min(NW, (left + 31) >> 5);
#pragma unroll
    for (int p = 0; p < 16; ++p) {
      if (p >= kw) break;
      unsigned key = 0;
      int ci = 0;
#pragma unroll
      for (int i = 0; i < RP; ++i) {
        const unsigned k = place[i] < 0 ? ((unsigned)__double2hiint(a[i][p]) & 0x7fffffffu) + 1 : 0;
        if (k > key) { key = k; ci = i; }
      }
      const unsigned best = __reduce_max_sync(0xffffffffu, key);
      const unsigned mine = __ballot_sync(0xffffffffu, key == best);
      if (best == 0 && lane == 0 && warp < nw) ckey[p & 1][warp] = 0;
      if (best > 0 && lane == __ffs(mine) - 1) {
        ckey[p & 1][warp] = best;
        cwho[p & 1][warp] = tid + ci * THREADS;
#pragma unroll
        for (int i = 0; i < RP; ++i)
          if (i == ci) {
            cinv[p & 1][warp] = 1.0 / a[i][p];
#pragma unroll
            for (int c = 0; c < 16; ++c)
              if (c >= p) cand[p & 1][warp][c] = a[i][c];
          }
      }
      __syncthreads();
      const unsigned wk = lane < nw ? ckey[p & 1][lane] : 0;
      const unsigned wbest = __reduce_max_sync(0xffffffffu, wk);
      const int w = __ffs(__ballot_sync(0xffffffffu, lane < nw && wk == wbest)) - 1;
      if (!NMC_DCHECK(w >= 0 && w < nw, 202)) break;
      const int piv = cwho[p & 1][w];
      const double ip = cinv[p & 1][w];
      if (tid == 0) {
        who[p] = piv;
        inv[k0 + p] = ip;
      }
      const double* pr = cand[p & 1][w];
      if (warp < nw) {
#pragma unroll
        for (int i = 0; i < RP; ++i) {
          if (piv == tid + i * THREADS) place[i] = p;
          const double l = place[i] < 0 ? a[i][p] * ip : 0.0;
          if (place[i] < 0) a[i][p] = l;
#pragma unroll
          for (int c = 0; c < 16; ++c)
            if (c > p) a[i][c] = fma(-l, pr[c], a[i][c]);
        }
      }
    }
    __syncthreads();
    // ------------------------------------------------- the new order; digits of the rows below
    for (int e = kw * 16 + tid; e < 256; e += THREADS) tri[e >> 4][e & 15] = 0.0;
    // pivot p moves to place k0 + p; the rows it displaces fill the places the pivots left
    const int wl = lane < kw ? who[lane] : 0;
    const unsigned taken = __reduce_or_sync(0xffffffffu, lane < kw && wl < kw ? 1u << wl : 0u);
    const unsigned outside = __ballot_sync(0xffffffffu, lane < kw && wl >= kw);
    const unsigned moved = ~taken & ((1u << kw) - 1);   // as many as `outside` has bits
#pragma unroll
    for (int i = 0; i < RP; ++i) {
      const int t = tid + i * THREADS;
      if (t >= left) continue;
      if (place[i] >= 0) {
        const int p = place[i];
        map[k0 + p] = row[i];   // (read by no one before the next barrier)
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          tri[p][c] = a[i][c];
          if (c >= p && c < kw) A[(long long)row[i] * lda + k0 + c] = a[i][c];   // U, for the way back
        }
      } else {
        int to = t;
        if (t < kw)
          to = who[__fns(outside, 0, __popc(moved & ((1u << t) - 1)) + 1)];
        if (!NMC_DCHECK(to >= kw && to < left, 203)) continue;
        map[k0 + to] = row[i];
        int E = Digits<double>::kExpMin;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
          a[i][c] = -a[i][c];
          E = max(E, Digits<double>::expo(a[i][c]));
        }
        re[to - kw] = Digits<double>::scale(E);
        cut16<double>(a[i], E, rd, to - kw, rs);
      }
    }
    __syncthreads();
    // ------------------------------------------------- the block's rows, and the update below
    const int c0 = k0 + kw;
    for (int c = c0 + tid; c < 2 * N; c += THREADS) {
      double x[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) x[q] = q < kw ? A[(long long)map[k0 + q] * lda + c] : 0.0;
#pragma unroll
      for (int s = 0; s < 16; ++s) {   // (tri is 0 beyond kw)
#pragma unroll
        for (int q = s + 1; q < 16; ++q) x[q] = fma(-tri[q][s], x[s], x[q]);
        if (s > 0 && s < kw) A[(long long)map[k0 + s] * lda + c] = x[s];
      }
    }
    __syncthreads();
    if (c0 >= N) break;
    for (int j0 = c0; j0 < 2 * N; j0 += chunk) {
      const int w = min(chunk, 2 * N - j0);
      cut_columns(j0, w, k0);
      __syncthreads();
      fold_tiles<double>([&](int r) { return A + (long long)map[c0 + r] * lda + j0; }, rda, rs, re, cda, cs, ce,
                         N - c0, w, (N & 1) == 0, warp, NW);
      __syncthreads();
    }
  }
  // ------------------------------------------------------------ upwards
  double* Yb = Y + (long long)b * NN;
  for (int k0 = (N - 1) & ~15; k0 >= 0; k0 -= 16) {
    const int kw = min(16, N - k0);
    for (int e = tid; e < 256; e += THREADS) {   // the block's U
      const int q = e >> 4, c = e & 15;
      tri[q][c] = q < kw && c < kw ? A[(long long)map[k0 + q] * lda + k0 + c] : 0.0;
    }
    for (int r = tid; r < k0; r += THREADS) {    // its columns in the rows above
      const double* src = A + (long long)map[r] * lda + k0;
      double u[16];
      int E = Digits<double>::kExpMin;
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        u[c] = c < kw ? -src[c] : 0.0;
        E = max(E, Digits<double>::expo(u[c]));
      }
      re[r] = Digits<double>::scale(E);
      cut16<double>(u, E, rd, r, rs);
    }
    __syncthreads();
    for (int c = tid; c < N; c += THREADS) {
      double x[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) x[q] = q < kw ? A[(long long)map[k0 + q] * lda + N + c] : 0.0;
#pragma unroll
      for (int s = 15; s >= 0; --s) {
        if (s >= kw) continue;
        x[s] *= inv[k0 + s];
#pragma unroll
        for (int q = 0; q < s; ++q) x[q] = fma(-tri[q][s], x[s], x[q]);
        Yb[(long long)(k0 + s) * N + c] = x[s];
        if (k0 > 0) A[(long long)map[k0 + s] * lda + N + c] = x[s];
      }
    }
    __syncthreads();
    if (k0 == 0) break;
    for (int j0 = 0; j0 < N; j0 += chunk) {
      const int w = min(chunk, N - j0);
      cut_columns(N + j0, w, k0);
      __syncthreads();
      fold_tiles<double>([&](int r) { return A + (long long)map[r] * lda + N + j0; }, rda, rs, re, cda, cs, ce,
                         k0, w, (N & 1) == 0, warp, NW);
      __syncthreads();
    }
  }
}

}  // namespace

// The lanes per column follow from N alone: as few as keep a lane's rows within 16 or 20 register
// pairs, and as many threads as columns need up to 512. Up to 64 sites a batch that fits the SMs at two
// (three) CTAs each takes the kernel with that many, which spills no registers, a larger one the kernel
// that puts four (five) there; the arithmetic is the same. us at two / four: 195 / 209 (64, 6), 426 / 338
// (64, 512); at three / five: 107 / 112 (36, 128). Up to 80 sites two are better than three either way:
// 275 / 305 (72, 6), 1137 / 1220 (72, 1024).
void qrp_udt(const double* X, double* U, double* D, double* Tp, double* ws, int N, int batch,
             cudaStream_t st) {
  auto run = [&](auto kernel, int LPC, int NB, int threads) {
    const int rows = 4 * NB * LPC;
    const size_t small = (qr_small_bytes(rows, N) + 15) & ~(size_t)15;
    const size_t big = qr_smem(LPC) ? (size_t)N * qr_ld(rows, LPC) * sizeof(long long) : 0;
    allow_max_dynamic_smem((const void*)kernel);
    kernel<<<batch, threads, small + big, st>>>(X, U, D, Tp, ws, N);
  };
  if (N <= 16) run(k_qrp<4, 1, 64, 4>, 4, 1, 64);
  else if (N <= 32) run(k_qrp<4, 2, 128, 4>, 4, 2, 128);
  else if (N <= 48 && batch > 3 * sm_count()) run(k_qrp<4, 3, 192, 5>, 4, 3, 192);
  else if (N <= 48) run(k_qrp<4, 3, 192, 3>, 4, 3, 192);
  else if (N <= 64 && batch > 2 * sm_count()) run(k_qrp<4, 4, 256, 4>, 4, 4, 256);
  else if (N <= 64) run(k_qrp<4, 4, 256, 2>, 4, 4, 256);
  else if (N <= 80) run(k_qrp<4, 5, 320, 2>, 4, 5, 320);
  else if (N <= 128) run(k_qrp<8, 4, 512, 1>, 8, 4, 512);
  else if (N <= 160) run(k_qrp<8, 5, 512, 1>, 8, 5, 512);
  else if (N <= 256) run(k_qrp<16, 4, 512, 1>, 16, 4, 512);
  else if (N <= 512) run(k_qrp<32, 4, 512, 1>, 32, 4, 512);
  else run(k_qrp<32, 8, 512, 1>, 32, 8, 512);
}

// (the threshold that the documented scratch sizes of nmc_green_noalloc follow)
bool stab_needs_workspace(int N) {
  const size_t small = ((size_t)N * 28 + 64 + 15) & ~(size_t)15;
  return small + 2 * (size_t)N * N * sizeof(double) > kSmemLimit;
}

void solve_stab(const double* X, const double* UR, long long sUR, const double* DR,
                long long sDR, double* Y, double* ws, int N, int batch, cudaStream_t st) {
  if (N <= kGaussJordanMax) {
    allow_max_dynamic_smem((const void*)k_solve_gj);
    k_solve_gj<<<batch, kSolveThreads, 2 * (size_t)N * N * sizeof(double), st>>>(X, UR, sUR, DR, sDR, Y, N);
    return;
  }
  // shared memory holds the augmented matrix wherever no workspace is promised
  const bool smem = !stab_needs_workspace(N);
  auto run = [&](auto kernel, int threads, size_t limit) {
    int lda = 2 * N;
    if (smem && (lda & 15) == 0 && N <= 96) lda += 8;   // rows 64 bytes apart modulo the banks
    const size_t big = smem ? (size_t)N * lda * sizeof(double) : 0;
    int chunk = 16;   // as many columns as there is room for
    while (chunk < 2 * N && big + solve_small_bytes(N, chunk + 16, threads / 32) <= limit) chunk += 16;
    const size_t bytes = big + solve_small_bytes(N, chunk, threads / 32);
    allow_max_dynamic_smem((const void*)kernel);
    kernel<<<batch, threads, bytes, st>>>(X, UR, sUR, DR, sDR, Y, ws, N, lda, chunk);
  };
  constexpr size_t kTwo = 113 * 1024, kOne = 227 * 1024;   // two CTAs to an SM (up to 72 sites they fit), or one
  if (N <= 72) run(k_solve<256, 1, 2, true>, 256, kTwo);
  else if (smem) run(k_solve<512, 1, 1, true>, 512, kOne);
  else if (N <= 512) run(k_solve<512, 1, 1, false>, 512, kOne);
  else run(k_solve<512, 2, 1, false>, 512, kOne);
}

NMC_DEBUG_READER(debug_fail_stab)

}  // namespace nmc
