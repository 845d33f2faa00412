// FP64-class batched products of two chain-private operands on the tensor cores.
//
// The FP64 pipe issues one warp multiply-add per 20 cycles and SM; a product of FP64 operands
// is cheaper as exact integer slices (Ozaki-style splitting; Ozaki, Ogita, Oishi, Rump, Numer.
// Algorithms 2012). Every row of op(A) and every column of op(B) is scaled by a power of two
// into 62-bit fixed point and cut into 7 balanced digits of 9 bits (|d| <= 256, exact in FP16).
// The 28 digit products s + t <= 6 accumulate in FP32, one accumulator per group g = s + t:
// over 64 terms the sums of groups 0..3 stay below 2^24 and are exact, those of groups 4..6
// (below 2^-36 of the product) as good as always. Longer sums are staged 48 terms at a time, and
// between two stages each accumulator's multiples of 512 move to the next group up, exactly (the
// first group's own sums stay below 2^24 up to K = 256). The groups are added up as 64-bit
// integers. An output's errors are then the digits' remainder (2^-62 of the row's and the
// column's maximum), the dropped groups (2^-62) and one rounding of a 63-bit sum -- below an
// FP64 chain of K roundings (measured on random operands, N = 64: 5e-17 of the result's norm
// against 2.4e-16). The sums' order depends on K alone, so a result does not depend on the
// batch or the tiling, which may follow the batch size.
//
// Why mma.sync and not tcgen05: both operands are private to a matrix of 16..144 rows, so a
// 128-row tcgen05 tile would hold several matrices and multiply each by the others' columns,
// and its accumulators would come back through tensor memory; the cutting and the epilogue,
// which are the same for both, already outweigh the tensor time (m16n8k16: 0.47 per cycle and
// SM, 12 us of 512 products of 64 x 64).
//
// One warp owns a 16 x 16 output block (7 groups x 8 accumulators per thread); a CTA is WM x WN
// warps (at most 8, two CTAs per SM), chosen at launch with the split of the rows and columns
// into equal parts, so that sizes that are no power of two waste little. All threads cut the
// tile's operands into shared memory first, eight entries of a row or column at a time.
#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>

#include "nmc_internal.cuh"

namespace nmc {

namespace {

NMC_DEBUG_FLAG

constexpr int kDigits = 7;
constexpr int kW = 9;                       // bits per digit
constexpr int kBits = 62;                   // |v| < 2^62
constexpr int kWhole = 64;                  // K staged at once up to here,
constexpr int kChunk = 48;                  // else this many terms at a time, with carries between
constexpr int kMaxFxK = 256;
constexpr int kMaxWarps = 8;
constexpr int kUnits = 3;                   // octets per thread held between scan and cut

struct FxTile {
  int WM, WN;       // warps
  int rm, rn;       // rows and columns per tile (<= 16 WM, 16 WN)
  int kc;           // staged terms at a time: K rounded up to 16, at most kChunk
};

__device__ __forceinline__ int biased_exp(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// v 2^k; a result outside the normal range goes through ldexp
__device__ __forceinline__ double scale_pow2(double v, int k) {
  const int e = biased_exp(v);
  if (e == 0) return v;   // v is a converted integer: only 0 has no exponent
  const int r = e + k;
  if (r >= 1 && r <= 2046) return __hiloint2double(__double2hiint(v) + k * (1 << 20), __double2loint(v));
  return ldexp(v, k);
}

// v as an FP32 pair, as df_from_double gives it, without the FP64 pipe's conversions: the 53-bit
// significand is cut at 24 bits (to nearest, ties to even), the signed rest is the low part.
// Outside the range where both parts are normal: df_from_double.
__device__ __forceinline__ df2 split_bits(double v) {
  const int h = __double2hiint(v);
  const unsigned l = (unsigned)__double2loint(v);
  const int e = ((h >> 20) & 0x7ff) - 1023;
  if (e < -70 || e > 126) return df_from_double(v);
  const unsigned top = (((unsigned)h & 0xfffffu) | 0x100000u) << 3 | (l >> 29);   // 24 bits
  const unsigned rest = l & 0x1fffffffu;                                          // 29 bits
  const unsigned up = (rest > 0x10000000u || (rest == 0x10000000u && (top & 1u))) ? 1u : 0u;
  const int low = (int)rest - (int)(up << 29);
  // a significand that rounds up to 2^24 carries into the exponent field
  const unsigned fb = ((unsigned)(e + 127) << 23) + ((top & 0x7fffffu) + up);
  const unsigned sgn = (unsigned)h & 0x80000000u;
  const float lo = (float)low * __uint_as_float((unsigned)(e - 52 + 127) << 23);
  return df2{__uint_as_float(fb | sgn), sgn ? -lo : lo};
}

__device__ __forceinline__ void ldmatrix4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

__device__ __forceinline__ void mma_f16(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                        unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// Eight entries of one vector (a row of op(A), a column of op(B)): terms k0 .. k0 + 7, zero past K
struct Octet {
  double x[8];
};
__device__ __forceinline__ void load8(Octet& o, const double* P, long long ks, int k0, int K,
                                      const double* brow) {
#pragma unroll
  for (int j = 0; j < 8; ++j) o.x[j] = k0 + j < K ? P[(k0 + j) * ks] : 0.0;
  if (brow) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (k0 + j < K) o.x[j] *= brow[k0 + j];
  }
}
__device__ __forceinline__ int max_exp(const Octet& o) {
  int m = 1;
#pragma unroll
  for (int j = 0; j < 8; ++j) m = max(m, biased_exp(o.x[j]));
  return m;
}

// Cut an octet into digits (most significant first), 16 bytes per digit at dst + s * stride.
// A significand left-aligned in 64 bits and shifted to the vector's scale is 62 bits; adding 256
// to every 9-bit field and reading the fields less 256 gives balanced digits. A field f in the
// low bits of FP16's 1024 + f, less 1280, is the digit; the sign goes in with the same
// multiply-add. Subnormals count as 0.
__device__ __forceinline__ void cut8(const Octet& o, int emax, unsigned char* dst, int stride) {
  unsigned w[kDigits][4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    unsigned long long u[2];
    unsigned short sg[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const double x = o.x[2 * p + q];
      const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
      const int e = (int)((h >> 20) & 0x7ffu);
      const unsigned mh = __funnelshift_l(l, h, 11) | 0x80000000u;
      const int sh = min(64 - kBits + emax - e, 63);
      u[q] = (((unsigned long long)mh << 32 | (l << 11)) >> sh) + 0x4020100804020100ull;
      sg[q] = e == 0 ? 0 : (unsigned short)(0x3c00u | ((h >> 16) & 0x8000u));   // 0 or +-1
    }
    const __half2 sgn = __halves2half2(__ushort_as_half(sg[0]), __ushort_as_half(sg[1]));
    const __half2 off = __hmul2(sgn, __float2half2_rn(-1280.f));
#pragma unroll
    for (int s = 0; s < kDigits; ++s) {
      const int bit = kW * (kDigits - 1 - s);
      const unsigned f0 = (unsigned)(u[0] >> bit), f1 = (unsigned)(u[1] >> bit);
      unsigned f = __byte_perm(f0, f1, 0x5410);   // the low halves of both
      if (s > 0) f &= 0x01ff01ffu;                // (the first digit's field may reach 512)
      f |= 0x64006400u;
      const __half2 d = __hfma2(*reinterpret_cast<__half2*>(&f), sgn, off);
      w[s][p] = *reinterpret_cast<const unsigned*>(&d);
    }
  }
#pragma unroll
  for (int s = 0; s < kDigits; ++s)
    *reinterpret_cast<uint4*>(dst + s * stride) = make_uint4(w[s][0], w[s][1], w[s][2], w[s][3]);
}

// MULTI: K > kChunk, the operands are staged chunk by chunk
template <bool MULTI>
__global__ void __launch_bounds__(kMaxWarps * 32, 2)
k_gemm_fx(const GemmArgs<double> g, const FxTile t) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int ev[2 * 16 * kMaxWarps];   // largest biased exponents: rows, then columns
  const int K = g.K, BM = 16 * t.WM, BN = 16 * t.WN;
  const int ldb = (t.kc + 8) * 2;          // bytes per staged vector: 16 B of padding
  const int sA = BM * ldb, sB = BN * ldb;  // bytes per digit
  unsigned char* As = smem;
  unsigned char* Bs = smem + kDigits * sA;
  const int b = blockIdx.z, tid = threadIdx.x, nthr = blockDim.x;
  const int m0 = blockIdx.y * t.rm, n0 = blockIdx.x * t.rn;
  const int mv = min(t.rm, g.M - m0), nv = min(t.rn, g.N - n0);
  const long long avs = g.transA ? 1 : g.lda, aks = g.transA ? g.lda : 1;
  const long long bvs = g.transB ? g.ldb : 1, bks = g.transB ? 1 : g.ldb;
  const double* A = g.A + (long long)b * g.sA + m0 * avs;
  const double* B = g.B + (long long)b * g.sB + n0 * bvs;

  double* br = (double*)(Bs + kDigits * sB);   // B's row scales
  const double* brow = g.brow.kind != SC_NONE ? br : nullptr;
  for (int v = tid; v < BM + BN; v += nthr) ev[v] = 1;
  if (brow)
    for (int k = tid; k < K; k += nthr) br[k] = scale_at(g.brow, b, k);
  __syncthreads();

  // unit e of a chunk of oc octets: the operand, vector and octet. Consecutive threads follow
  // the index that is contiguous in memory.
  auto unit = [&](int e, int oc, int& v, int& o, bool& isb) {
    isb = e >= mv * oc;
    if (isb) e -= mv * oc;
    const int n = isb ? nv : mv;
    if ((isb ? bks : aks) == 1) { v = e / oc; o = e - v * oc; } else { o = e / n; v = e - o * n; }
  };
  auto load = [&](Octet& x, int v, int o, bool isb, int k0) {
    if (isb) load8(x, B + v * bvs, bks, k0 + 8 * o, K, brow);
    else load8(x, A + v * avs, aks, k0 + 8 * o, K, nullptr);
  };
  auto cut = [&](const Octet& x, int v, int o, bool isb) {
    if (!NMC_DCHECK(v < (isb ? BN : BM) && 8 * o + 8 <= t.kc, 412)) return;
    if (isb) cut8(x, ev[BM + v], Bs + v * ldb + o * 16, sB);
    else cut8(x, ev[v], As + v * ldb + o * 16, sA);
  };

  const int warp = tid >> 5, lane = tid & 31;
  const int wm = warp / t.WN, wn = warp - wm * t.WN;
  const int all = (K + 7) / 8 * (mv + nv);   // units of the whole operands
  if (MULTI) {
    const int oc = (K + 7) / 8;
    for (int e = tid; e < all; e += nthr) {
      int v, o; bool isb;
      unit(e, oc, v, o, isb);
      Octet x;
      load(x, v, o, isb, 0);
      atomicMax(&ev[(isb ? BM : 0) + v], max_exp(x));
    }
    __syncthreads();
  }

  float acc[kDigits][2][4];
  // H = groups 0..2, L = groups 3..6 of output i as integers: value (H 2^36 + L) 2^54
  auto sums = [&](int i, long long& H, long long& L) {
    const int nt = i >> 2, w = i & 3;
    int q[kDigits];
#pragma unroll
    for (int s = 0; s < kDigits; ++s) q[s] = __float2int_rn(acc[s][nt][w]);
    H = (long long)q[0] * (1 << 18) + ((long long)q[1] * (1 << 9) + q[2]);
    L = (long long)q[3] * (1 << 27) + ((long long)q[4] * (1 << 18) + ((long long)q[5] * (1 << 9) + q[6]));
  };

#pragma unroll
  for (int s = 0; s < kDigits; ++s)
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[s][i >> 2][i & 3] = 0.f;
  for (int k0 = 0; k0 < K; k0 += t.kc) {
    const int kn = min(t.kc, K - k0), kp = (kn + 15) & ~15, oc = kp / 8;
    const int n = oc * (mv + nv);
    if (!MULTI) {   // scan and cut from registers
      Octet x[kUnits];
      int v[kUnits], o[kUnits];
      bool isb[kUnits];
#pragma unroll
      for (int i = 0; i < kUnits; ++i) {
        const int e = tid + i * nthr;
        if (e >= n) continue;
        unit(e, oc, v[i], o[i], isb[i]);
        load(x[i], v[i], o[i], isb[i], 0);
      }
#pragma unroll
      for (int i = 0; i < kUnits; ++i)
        if (tid + i * nthr < n) atomicMax(&ev[(isb[i] ? BM : 0) + v[i]], max_exp(x[i]));
      for (int e = tid + kUnits * nthr; e < n; e += nthr) {   // (few threads, a wide tile)
        int v1, o1; bool b1;
        unit(e, oc, v1, o1, b1);
        Octet y;
        load(y, v1, o1, b1, 0);
        atomicMax(&ev[(b1 ? BM : 0) + v1], max_exp(y));
      }
      __syncthreads();
      for (int e = tid + kUnits * nthr; e < n; e += nthr) {
        int v1, o1; bool b1;
        unit(e, oc, v1, o1, b1);
        Octet y;
        load(y, v1, o1, b1, 0);
        cut(y, v1, o1, b1);
      }
#pragma unroll
      for (int i = 0; i < kUnits; ++i)
        if (tid + i * nthr < n) cut(x[i], v[i], o[i], isb[i]);
    } else {
      for (int e = tid; e < n; e += nthr) {
        int v, o; bool isb;
        unit(e, oc, v, o, isb);
        Octet x;
        load(x, v, o, isb, k0);
        cut(x, v, o, isb);
      }
    }
    __syncthreads();

    const unsigned pa = (unsigned)__cvta_generic_to_shared(As) + (wm * 16 + (lane & 15)) * ldb +
                        (lane >> 4) * 16;
    const unsigned pb = (unsigned)__cvta_generic_to_shared(Bs) +
                        (wn * 16 + (lane & 7) + ((lane >> 4) & 1) * 8) * ldb + ((lane >> 3) & 1) * 16;
#pragma unroll 1
    for (int k = 0; k < kp; k += 16) {
      unsigned bf[kDigits][4];
#pragma unroll
      for (int s = 0; s < kDigits; ++s) ldmatrix4(bf[s], pb + s * sB + k * 2);
#pragma unroll
      for (int s = 0; s < kDigits; ++s) {
        unsigned af[4];
        ldmatrix4(af, pa + s * sA + k * 2);
#pragma unroll
        for (int q = 0; q + s < kDigits; ++q) {
          mma_f16(acc[s + q][0], af, bf[q][0], bf[q][1]);
          mma_f16(acc[s + q][1], af, bf[q][2], bf[q][3]);
        }
      }
    }
    if (MULTI && k0 + t.kc < K) {   // carries: multiples of 512 to the next group up
      constexpr float kM = 12582912.f;   // 1.5 2^23: adding and removing it rounds to an integer
#pragma unroll
      for (int s = kDigits - 1; s > 0; --s)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          float& a = acc[s][i >> 2][i & 3];
          const float c = __fsub_rn(__fmaf_rn(a, 1.f / 512.f, kM), kM);
          a = __fmaf_rn(c, -512.f, a);
          acc[s - 1][i >> 2][i & 3] += c;
        }
      __syncthreads();   // the next chunk overwrites the digits
    }
  }

  // the output scales, in the place of the digits
  const bool rscale = g.crow.kind != SC_NONE;
  const bool cscale = g.ccol.kind != SC_NONE || g.bcol.kind != SC_NONE;
  double* rs = (double*)smem;
  double* cs = rs + BM;
  if (rscale || cscale) {
    __syncthreads();
    if (rscale)
      for (int i = tid; i < mv; i += nthr) rs[i] = scale_at(g.crow, b, m0 + i);
    if (cscale)
      for (int j = tid; j < nv; j += nthr) {
        double c = g.ccol.kind != SC_NONE ? scale_at(g.ccol, b, n0 + j) : 1.0;
        if (g.bcol.kind != SC_NONE) c *= scale_at(g.bcol, b, n0 + j);
        cs[j] = c;
      }
    __syncthreads();
  }

  long long dmax = 0;   // bits of the largest |C - ref| (a NaN's order above every number's)
  double far_out = 0.0, far_ref = 0.0;   // FP32-pair reference: the entry that is furthest off
  float far = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = wm * 16 + (lane >> 2) + ((i >> 1) & 1) * 8;
    const int c = wn * 16 + (i >> 2) * 8 + (lane & 3) * 2 + (i & 1);
    if (r >= mv || c >= nv) continue;
    long long H, L;
    sums(i, H, L);
    // (H 2^36 + L) 2^54: the 63 leading bits, rounded once
    H += L >> 36;
    L &= (1ll << 36) - 1;
    const int s = min(__clzll(H ^ (H >> 63)) - 1, 36);
    const long long V = (H << s) + (L >> (36 - s));
    const int ea = ev[r], eb = ev[BM + c];
    double v = scale_pow2((double)V, ea + eb - 2 * (1022 + kBits) + 54 + 36 - s);
    if (ea == 0x7ff || eb == 0x7ff) v = __longlong_as_double(0x7ff8000000000000ll);
    if (rscale) v *= rs[r];
    if (cscale) v *= cs[c];
    const int gm = m0 + r, gn = n0 + c;
    if (!NMC_DCHECK(gm < g.M && gn < g.N, 411)) continue;
    if (g.Cin) v += g.beta * g.Cin[(long long)b * g.sCin + (long long)gm * g.ldcin + gn];
    const long long idx = (long long)gm * g.ldc + gn;
    df2 p{0.f, 0.f};
    if (g.Cdf || g.ref_is_float == 2) p = split_bits(v);
    if (g.ref) {
      const long long ri = (long long)b * g.sRef + idx;
      if (g.ref_is_float == 2) {
        const df2 q = ((const df2*)g.ref)[ri];
        const float d = fabsf((p.hi - q.hi) + (p.lo - q.lo));
        if (!(d <= far) && far == far)   // larger, or the first NaN
          far = d, far_out = v, far_ref = (double)q.hi + (double)q.lo;
      } else {
        const double q = g.ref_is_float == 1 ? (double)((const float*)g.ref)[ri]
                                             : ((const double*)g.ref)[ri];
        dmax = max(dmax, __double_as_longlong(fabs(v - q)));
      }
    }
    g.C[(long long)b * g.sC + idx] = v;
    if (g.Cf) g.Cf[(long long)b * g.sCf + idx] = (float)v;
    if (g.Cdf) g.Cdf[(long long)b * g.sCdf + idx] = p;
  }
  if (g.drift) {
    if (g.ref_is_float == 2) dmax = __double_as_longlong(fabs(far_out - far_ref));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    if (lane == 0 && dmax != 0)
      atomicMax(g.drift + (g.ns == 2 ? b >> 1 : b), (unsigned long long)dmax);
  }
}

int up_div(int a, int b) { return (a + b - 1) / b; }

// The split of the rows and columns: over all splits whose blocks fit kMaxWarps warps, the least
// of an estimate of the time per SM, in cycles -- cutting ~8 instructions' issue per entry
// quarter-warp, a warp's 16 terms 120 cycles of the tensor pipe, an output ~19 instructions
// per warp and cycle share -- or, for a batch that leaves SMs idle, of one CTA's own latency.
FxTile fx_tile(const GemmArgs<double>& g) {
  const int sms = sm_count();
  FxTile best{};
  double best_cost = 1e300;
  for (int tm = 1; tm <= up_div(g.M, 16); ++tm)
    for (int tn = 1; tn <= up_div(g.N, 16); ++tn) {
      FxTile t;
      t.rm = up_div(g.M, tm);
      t.rn = up_div(g.N, tn);
      t.WM = up_div(t.rm, 16);
      t.WN = up_div(t.rn, 16);
      const int warps = t.WM * t.WN;
      if (warps > kMaxWarps || up_div(g.M, t.rm) != tm || up_div(g.N, t.rn) != tn) continue;
      const double k16 = up_div(g.K, 16);
      const double cut = (double)(t.rm + t.rn) * g.K * 0.26 * (g.K > kWhole ? 1.3 : 1.0);
      const double work = cut + warps * k16 * 120 * 0.7 + warps * 256 * 0.6;
      const double alone = 3000 + cut * 4 / (warps < 4 ? warps : 4) + k16 * 56 * 9;
      const double ctas = (double)tm * tn * g.batch;
      const double per_sm = std::ceil(ctas / sms);
      const double cost = std::fmax(per_sm * work, std::ceil(per_sm / 2) * alone);
      if (cost < best_cost) best_cost = cost, best = t;
    }
  best.kc = g.K > kWhole ? kChunk : (g.K + 15) & ~15;
  return best;
}

template <bool MULTI>
void run_fx(const GemmArgs<double>& g, const FxTile& t, cudaStream_t st) {
  const int BM = 16 * t.WM, BN = 16 * t.WN;
  size_t bytes = (size_t)kDigits * (BM + BN) * (t.kc + 8) * 2;
  bytes = std::max(bytes, sizeof(double) * (size_t)(BM + BN));   // the scales share its place
  if (g.brow.kind != SC_NONE) bytes += (size_t)g.K * sizeof(double);
  allow_max_dynamic_smem((const void*)k_gemm_fx<MULTI>);
  k_gemm_fx<MULTI><<<dim3(up_div(g.N, t.rn), up_div(g.M, t.rm), g.batch), 32 * t.WM * t.WN,
                     bytes, st>>>(g, t);
}

}  // namespace

bool gemm_fx_supported(const GemmArgs<double>& g) { return g.K <= kMaxFxK; }

void gemm_fx(const GemmArgs<double>& g, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0 || g.batch <= 0) return;
  const FxTile t = fx_tile(g);
  if (g.K > kWhole) run_fx<true>(g, t, st);
  else run_fx<false>(g, t, st);
}

NMC_DEBUG_READER(debug_fail_gemm_fx)

}  // namespace nmc
