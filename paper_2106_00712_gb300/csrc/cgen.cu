// Convolutional field generator (include/nmc_cgen.h): four periodic 3D convolutions
// (3 x 3 x 3 kernels, channels 1 -> C -> C -> C -> 1, ReLU between) mapping N(0,1) noise
// to Bernoulli logits per field entry, trained by maximum likelihood on DQMC fields.
//
// Every convolution reads BF16 operands and accumulates in FP32 (SIMT FMA): the activations
// and the gradients flowing between layers are stored as BF16, the weights are used as a
// BF16 copy of the FP32 master weights. Kernels, all over the batch [n][C][S] with
// S = L_tau * Ly * Lx (x fastest, so the last layer's entry p is field entry (i, l) at
// p = l N + i):
//   k_cg_conv    out[n][co][p] = b[co] + sum_k sum_ci W[co][ci][k] in[n][ci][p + d_k], then
//                ReLU and BF16, or FP32 logits for the last layer; the same kernel with -d_k
//                is the backward convolution into the inputs;
//   k_cg_loss    the Bernoulli negative log-likelihood and dL/dlogit = (sigmoid(l) - y) /
//                (n S), as BF16 for the backward convolutions;
//   k_cg_conv    dL/din[n][ci][q] = sum_k sum_co W[co][ci][k] g[n][co][q - d_k], times the
//                ReLU mask of that input (it is the previous layer's output), as BF16;
//   k_cg_bwd_w_tc dL/dW[co][ci][k] = sum_{n,p} g[n][co][p] in[n][ci][p + d_k] and
//                dL/db[co] = sum g[n][co][p], as one product over all positions;
//   k_cg_fwd, k_cg_bwd_in, k_cg_bwd_w: the same one output per thread (or CTA), for small calls and
//                shapes whose halo does not fit shared memory or whose rows have odd length;
//   k_cg_adam    Adam on the FP32 master weights, then their BF16 copy.
// Noise and Bernoulli draws are Philox4x32-10 words (counter (p, sample, stream, tag)).
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <string>
#include <type_traits>
#include <vector>

#include "nmc_cgen.h"
#include "nmc_internal.cuh"

using nmc::philox4x32_10;

namespace {

constexpr int kLayers = 4;
constexpr int kK = 27;             // 3 x 3 x 3 kernel entries
constexpr uint32_t kTagNoise = 5u, kTagDraw = 6u, kTagInit = 7u;
constexpr int kFwdThreads = 128;
constexpr int kWThreads = 256;

struct Dims {
  int T, A, B;   // L_tau, Ly, Lx
  __host__ __device__ int S() const { return T * A * B; }
};

__device__ __forceinline__ float bf(__nv_bfloat16 v) { return __bfloat162float(v); }

// entry p + d_k (periodic), d_k = (k / 9 - 1, (k / 3) % 3 - 1, k % 3 - 1)
__device__ __forceinline__ int neighbour(const Dims& d, int t, int a, int b, int k, int sign) {
  const int dt = sign * (k / 9 - 1), da = sign * ((k / 3) % 3 - 1), db = sign * (k % 3 - 1);
  int tt = t + dt, aa = a + da, bb = b + db;
  tt += tt < 0 ? d.T : tt >= d.T ? -d.T : 0;
  aa += aa < 0 ? d.A : aa >= d.A ? -d.A : 0;
  bb += bb < 0 ? d.B : bb >= d.B ? -d.B : 0;
  return (tt * d.A + aa) * d.B + bb;
}

__global__ void k_cg_fwd(const __nv_bfloat16* __restrict__ in, int Cin,
                         const __nv_bfloat16* __restrict__ W, const float* __restrict__ bias,
                         int Cout, Dims d, int relu, __nv_bfloat16* __restrict__ out_h,
                         float* __restrict__ out_f) {
  extern __shared__ float sw[];   // [Cin][27] of output channel co
  const int co = blockIdx.y, n = blockIdx.z, S = d.S();
  for (int e = threadIdx.x; e < Cin * kK; e += blockDim.x) sw[e] = bf(W[(long long)co * Cin * kK + e]);
  __syncthreads();
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= S) return;
  const int t = p / (d.A * d.B), rem = p - t * d.A * d.B, a = rem / d.B, b = rem - a * d.B;
  const __nv_bfloat16* x = in + (long long)n * Cin * S;
  float acc = bias[co];
  for (int k = 0; k < kK; ++k) {
    const int q = neighbour(d, t, a, b, k, 1);
    for (int ci = 0; ci < Cin; ++ci) acc = fmaf(sw[ci * kK + k], bf(x[(long long)ci * S + q]), acc);
  }
  if (relu) out_h[((long long)n * Cout + co) * S + p] = __float2bfloat16_rn(fmaxf(acc, 0.f));
  else out_f[((long long)n * Cout + co) * S + p] = acc;
}

__global__ void k_cg_loss(const float* __restrict__ logits, const int8_t* __restrict__ fields,
                          long long total, float inv_count, __nv_bfloat16* __restrict__ g,
                          double* __restrict__ loss_sum) {
  __shared__ double red[kWThreads / 32];
  double part = 0.0;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const float l = logits[e];
    const float y = fields[e] > 0 ? 1.f : 0.f;
    // softplus(l) - y l, with softplus(l) = max(l, 0) + log1p(exp(-|l|))
    part += (double)(fmaxf(l, 0.f) + log1pf(expf(-fabsf(l))) - y * l);
    const float sg = 1.f / (1.f + expf(-l));
    g[e] = __float2bfloat16_rn((sg - y) * inv_count);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += red[w];
    atomicAdd(loss_sum, s);
  }
}

__global__ void k_cg_bwd_in(const __nv_bfloat16* __restrict__ g, int Cout,
                            const __nv_bfloat16* __restrict__ W, int Cin, Dims d,
                            const __nv_bfloat16* __restrict__ act, __nv_bfloat16* __restrict__ gin) {
  extern __shared__ float sw[];   // [Cout][27] of input channel ci
  const int ci = blockIdx.y, n = blockIdx.z, S = d.S();
  for (int e = threadIdx.x; e < Cout * kK; e += blockDim.x) {
    const int co = e / kK, k = e - co * kK;
    sw[e] = bf(W[((long long)co * Cin + ci) * kK + k]);
  }
  __syncthreads();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= S) return;
  const long long o = ((long long)n * Cin + ci) * S + q;
  if (!(bf(act[o]) > 0.f)) {   // the ReLU's derivative is 0 there
    gin[o] = __float2bfloat16_rn(0.f);
    return;
  }
  const int t = q / (d.A * d.B), rem = q - t * d.A * d.B, a = rem / d.B, b = rem - a * d.B;
  const __nv_bfloat16* gg = g + (long long)n * Cout * S;
  float acc = 0.f;
  for (int k = 0; k < kK; ++k) {
    const int p = neighbour(d, t, a, b, k, -1);   // q - d_k
    for (int co = 0; co < Cout; ++co) acc = fmaf(sw[co * kK + k], bf(gg[(long long)co * S + p]), acc);
  }
  gin[o] = __float2bfloat16_rn(acc);
}

__global__ void __launch_bounds__(kWThreads)
k_cg_bwd_w(const __nv_bfloat16* __restrict__ g, int Cout, const __nv_bfloat16* __restrict__ h,
           int Cin, Dims d, int n, float* __restrict__ gW, float* __restrict__ gb) {
  __shared__ float red[kWThreads / 32][kK + 1];
  const int ci = blockIdx.x, co = blockIdx.y, S = d.S();
  float acc[kK + 1];
#pragma unroll
  for (int k = 0; k <= kK; ++k) acc[k] = 0.f;
  const long long total = (long long)n * S;
  for (long long e = threadIdx.x; e < total; e += blockDim.x) {
    const int s = (int)(e / S), p = (int)(e - (long long)s * S);
    const float gv = bf(g[((long long)s * Cout + co) * S + p]);
    if (gv == 0.f) continue;
    const int t = p / (d.A * d.B), rem = p - t * d.A * d.B, a = rem / d.B, b = rem - a * d.B;
    const __nv_bfloat16* x = h + ((long long)s * Cin + ci) * S;
#pragma unroll
    for (int k = 0; k < kK; ++k) acc[k] = fmaf(gv, bf(x[neighbour(d, t, a, b, k, 1)]), acc[k]);
    acc[kK] += gv;
  }
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k <= kK; ++k) {
    float v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x <= kK) {
    float s = 0.f;
    for (int w = 0; w < kWThreads / 32; ++w) s += red[w][threadIdx.x];
    if (threadIdx.x < kK) gW[((long long)co * Cin + ci) * kK + threadIdx.x] = s;
    else if (ci == 0) gb[co] = s;
  }
}

// ---------------------------------------------------------------------------- tiled convolution
// One CTA (4 warps): PT consecutive positions of one sample x up to 32 output channels. The
// tile's slices of the input, with a periodic halo of one in every axis, sit in shared memory
// as words of two channels, so a neighbour is a constant word offset. A thread owns TP positions
// (32 apart, so a warp reads consecutive words) x 8 channels (TC = 8; 2 for a single output
// channel), accumulated in the order k, then input channel -- one fused multiply-add per term,
// as one output per thread would, so every output has the same bits whatever the tile -- with
// two channels per packed FP32 instruction (fma.rn.f32x2: 3.68 multiply-adds per cycle and SM
// against 3.45 for scalar ones, at half the issue slots). Weights come as FP32 [k][Cin][CoP]
// rows, the three k of one (t, y) neighbour per stage, the next stage in flight.
// What bounds it: the FP32 pipe (9.1 G multiply-adds of a 64 x 40 x 8 x 8 batch's two middle
// layers: 270 us at the packed rate). Measured per middle layer of that batch: 1064 us with one
// output per thread (one load per multiply-add), 256 now (one k per
// stage, which lets four CTAs on an SM instead of three: 262).
enum ConvMode { kHidden, kLogits, kBackward };
constexpr int kConvThreads = 128;

__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a,
                                     unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ int wrap1(int i, int n) { return i < 0 ? i + n : i >= n ? i - n : i; }

template <int TP, int TC, int MODE>
__global__ void __launch_bounds__(kConvThreads)
k_cg_conv(const __nv_bfloat16* __restrict__ in, int Cin, const float* __restrict__ wt, int CoP,
          const float* __restrict__ bias, int Cout, Dims d, int wco,
          const __nv_bfloat16* __restrict__ act, __nv_bfloat16* __restrict__ out_h,
          float* __restrict__ out_f) {
  extern __shared__ __align__(16) unsigned smc[];
  const int S = d.S(), AB = d.A * d.B, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wp = kConvThreads / 32 / wco;          // warps along the positions
  const int PT = wp * 32 * TP, p0 = blockIdx.x * PT, n = blockIdx.z;
  const int pe = min(p0 + PT, S) - 1;              // last position
  const int t_first = p0 / AB, ns = pe / AB - t_first + 3;
  const int PB = d.B + 2, PS = (d.A + 2) * PB, PW = ns * PS;
  const int pairs = (Cin + 1) >> 1, cos = TC * wco;  // output channels of this CTA
  const int co0 = blockIdx.y * cos;
  unsigned* X = smc;                               // [pairs][PW]
  float* W = (float*)(X + ((pairs * PW + 3) & ~3));  // [2][3][Cin][cos]
  const int wsz = 3 * Cin * cos;

  // stage c, the three k of the (t, y) neighbour c: rows of cos floats (16-byte pieces; 8 for TC = 2)
  auto fetch = [&](int c) {
    constexpr int V = TC == 8 ? 4 : 2;
    const int pieces = 3 * Cin * (cos / V);
    float* dst = W + (c & 1) * wsz;
    for (int e = tid; e < pieces; e += kConvThreads) {
      const int row = e / (cos / V), q = (e - row * (cos / V)) * V;
      if (co0 + q >= CoP) continue;
      const float* src = wt + ((long long)c * 3 * Cin + row) * CoP + co0 + q;
      const unsigned a = (unsigned)__cvta_generic_to_shared(dst + row * cos + q);
      if (V == 4) asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(a), "l"(src) : "memory");
      else asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(a), "l"(src) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0);

  const __nv_bfloat16* x = in + (long long)n * Cin * S;
  for (int q = tid; q < PW; q += kConvThreads) {
    const int sl = q / PS, r = q - sl * PS, ar = r / PB, br = r - ar * PB;
    const int src = (wrap1(t_first - 1 + sl, d.T) * d.A + wrap1(ar - 1, d.A)) * d.B + wrap1(br - 1, d.B);
    const unsigned short* xs = reinterpret_cast<const unsigned short*>(x) + src;
#pragma unroll 4
    for (int c = 0; c < pairs; ++c) {
      const unsigned lo = xs[(long long)(2 * c) * S];
      const unsigned hi = 2 * c + 1 < Cin ? xs[(long long)(2 * c + 1) * S] : 0u;
      X[c * PW + q] = lo | hi << 16;
    }
  }

  const int cg = warp % wco, co = co0 + cg * TC;   // this thread's first output channel
  const int pt = p0 + (warp / wco) * 32 * TP + lane;
  int base[TP];
#pragma unroll
  for (int j = 0; j < TP; ++j) {
    const int p = min(pt + 32 * j, pe);            // (past the tile: any position, not stored)
    const int t = p / AB, r = p - t * AB, a = r / d.B, b = r - a * d.B;
    base[j] = ((t - t_first + 1) * (d.A + 2) + a + 1) * PB + b + 1;
  }
  unsigned long long acc[TP][TC / 2];
#pragma unroll
  for (int c = 0; c < TC / 2; ++c) {
    const float b0 = MODE != kBackward && co + 2 * c < Cout ? bias[co + 2 * c] : 0.f;
    const float b1 = MODE != kBackward && co + 2 * c + 1 < Cout ? bias[co + 2 * c + 1] : 0.f;
#pragma unroll
    for (int j = 0; j < TP; ++j) acc[j][c] = pack2(b0, b1);
  }
  constexpr int kSign = MODE == kBackward ? -1 : 1;
  auto terms = [&](const float (&v)[TP], const float* w) {
    unsigned long long wv[TC / 2];
    if constexpr (TC == 8) {
      const ulonglong2 u0 = *reinterpret_cast<const ulonglong2*>(w);
      const ulonglong2 u1 = *reinterpret_cast<const ulonglong2*>(w + 4);
      wv[0] = u0.x; wv[1] = u0.y; wv[2] = u1.x; wv[3] = u1.y;
    } else {
      wv[0] = *reinterpret_cast<const unsigned long long*>(w);
    }
#pragma unroll
    for (int j = 0; j < TP; ++j) {
      const unsigned long long vv = pack2(v[j], v[j]);
#pragma unroll
      for (int q = 0; q < TC / 2; ++q) fma2(acc[j][q], wv[q], vv);
    }
  };
  for (int c = 0; c < 9; ++c) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();              // stage c is here, stage c - 1 is read
    if (c + 1 < 9) fetch(c + 1);
    const int row = kSign * ((c / 3 - 1) * PS + (c % 3 - 1) * PB);
#pragma unroll 1
    for (int db = 0; db < 3; ++db) {
      const unsigned* Xk = X + row + kSign * (db - 1);
      const float* Wk = W + (c & 1) * wsz + db * Cin * cos + cg * TC;
#pragma unroll 2
      for (int ci = 0; ci < Cin; ci += 2, Xk += PW, Wk += 2 * cos) {
        float lo[TP], hi[TP];
#pragma unroll
        for (int j = 0; j < TP; ++j) {
          const unsigned u = Xk[base[j]];
          lo[j] = __uint_as_float(u << 16);
          hi[j] = __uint_as_float(u & 0xffff0000u);
        }
        terms(lo, Wk);
        if (ci + 1 < Cin) terms(hi, Wk + cos);
      }
    }
  }

#pragma unroll
  for (int j = 0; j < TP; ++j) {
    const int p = pt + 32 * j;
    if (p > pe) continue;
#pragma unroll
    for (int c = 0; c < TC; ++c) {
      if (co + c >= Cout) continue;
      const unsigned long long u = acc[j][c / 2];
      const float v = __uint_as_float((unsigned)(c & 1 ? u >> 32 : u));
      const long long o = ((long long)n * Cout + co + c) * S + p;
      if (MODE == kLogits) out_f[o] = v;
      else if (MODE == kHidden) out_h[o] = __float2bfloat16_rn(fmaxf(v, 0.f));
      else out_h[o] = __float2bfloat16_rn(bf(act[o]) > 0.f ? v : 0.f);   // the ReLU's derivative
    }
  }
}

// FP32 copies of the layers' BF16 weights as k_cg_conv reads them, a layer per blockIdx.y: wf
// [k][Cin][CoP], wb [k][Cout][CiP] (the padding zero)
struct LayoutArgs {
  const __nv_bfloat16* W[kLayers];
  float *wf[kLayers], *wb[kLayers];
  int cin[kLayers], cout[kLayers];
};
__host__ __device__ constexpr int pad8(int c) { return (c + 7) & ~7; }

__global__ void k_cg_layout(LayoutArgs a) {
  const int j = blockIdx.y, Cin = a.cin[j], Cout = a.cout[j], CoP = pad8(Cout), CiP = pad8(Cin);
  const __nv_bfloat16* W = a.W[j];
  float *wf = a.wf[j], *wb = a.wb[j];
  const int nf = kK * Cin * CoP, total = nf + kK * Cout * CiP;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    const bool f = e < nf;
    const int r = f ? e : e - nf, P = f ? CoP : CiP, C = f ? Cin : Cout;
    const int k = r / (C * P), u = r / P - k * C, v = r % P;   // u: summed channel, v: output
    const int ci = f ? u : v, co = f ? v : u;
    (f ? wf : wb)[r] = ci < Cin && co < Cout ? bf(W[((long long)co * Cin + ci) * kK + k]) : 0.f;
  }
}

// ---------------------------------------------------------------------------- weight gradients
// gW[co][ci][k] = sum over all positions of g[co][p] h[ci][p + d_k]: one product with M = co,
// N = (k, ci), K = positions, BF16 operands and FP32 sums, mma.sync m16n8k16. A persistent CTA of
// nine warps, one per (t, y) neighbour, holds all 27 Cin Cout sums; per tile of TT slices of one
// sample it stages g [co][position] and h three times, shifted by -1, 0, 1 along x, with a
// halo in t and y, so that a warp's B operand (pairs of consecutive positions) is a 4-byte read
// at a constant offset. The tensor core cuts the low bits of its sums, so it adds 32 positions at a time
// only: their sums are added in registers (FP32, to nearest), a tile's in shared memory, and the CTAs'
// in a fixed order with the rounding errors carried along (k_cg_sum; how the tiles are shared out, and so
// the last bits, follow the SM count).
// What bounds it: staging (the product itself is 9.1 GFLOP per middle layer, 20 us). Measured per
// middle layer at batch 64 x 40 x 8 x 8, 32 channels: 3105 us with one CTA per (ci, co), 108 with a tile's
// 512 positions left to the tensor core and the CTAs' sums added one after the other. Errors were then up to
// 1.4e-6 of a layer's largest entry (1e-7 to 3e-7 rms), with one CTA per (ci, co) 1.9e-7 (2e-8), now 8e-8
// (1e-8); the whole gradient call takes 1542 us instead of 1522 (16 positions at a time: 7e-8, 1561).
constexpr int kBwThreads = 288;

__device__ __forceinline__ void mma_bf(float (&d)[4], const unsigned (&a)[4], unsigned b0,
                                       unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// acc += a b over K steps of 16 terms: the tensor core sums these, the addition rounds to nearest
template <int K>
__device__ __forceinline__ void add_products(float (&acc)[4], const unsigned (&a)[K][4], const unsigned (&b)[K][2]) {
  float d[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int k = 0; k < K; ++k) mma_bf(d, a[k], b[k][0], b[k][1]);
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i] = __fadd_rn(acc[i], d[i]);
}

struct BwTile {
  int TT, ABp;     // slices per tile; positions per slice, padded to 16
  int gld;         // BF16 per row of g
  int hld;         // BF16 per channel of one shifted copy of h
  int per_sample, total;
};

template <int MT, int NC>
__global__ void __launch_bounds__(kBwThreads)
k_cg_bwd_w_tc(const __nv_bfloat16* __restrict__ g, int Cout, const __nv_bfloat16* __restrict__ h,
              int Cin, Dims d, BwTile t, float* __restrict__ part, int P) {
  constexpr int kAcc = MT * 3 * NC * 4 + MT * 4;   // sums per thread (the last MT * 4: biases)
  extern __shared__ __align__(16) unsigned char smb[];
  float* sums = (float*)smb;                                 // [kAcc][kBwThreads]
  __nv_bfloat16* Gs = (__nv_bfloat16*)(sums + kAcc * kBwThreads);   // [MT 16][gld]
  __nv_bfloat16* Hs = Gs + MT * 16 * t.gld;                  // [3][NC 8][hld]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int S = d.S(), AB = d.A * d.B, A2 = d.A + 2;
  const int dt = warp / 3 - 1, da = warp % 3 - 1;
  for (int i = 0; i < kAcc; ++i) sums[i * kBwThreads + tid] = 0.f;

  for (int tile = blockIdx.x; tile < t.total; tile += gridDim.x) {
    const int s = tile / t.per_sample, t0 = (tile - s * t.per_sample) * t.TT;
    __syncthreads();
    // g: pairs of positions, zero past the slice, the sample and Cout
    const int gw = t.TT * t.ABp / 2;
    for (int e = tid; e < MT * 16 * gw; e += kBwThreads) {
      const int co = e / gw, w = 2 * (e - co * gw), ts = w / t.ABp, q = w - ts * t.ABp;
      unsigned v = 0u;
      if (co < Cout && t0 + ts < d.T && q < AB)
        v = *reinterpret_cast<const unsigned*>(g + ((long long)s * Cout + co) * S + (t0 + ts) * AB + q);
      *reinterpret_cast<unsigned*>(Gs + co * t.gld + w) = v;
    }
    // h: a row of B entries per thread, and its two shifts
    const int rows = (t.TT + 2) * A2, copy = NC * 8 * t.hld;
    for (int e = tid; e < NC * 8 * rows; e += kBwThreads) {
      const int ci = e / rows, r = e - ci * rows, ts = r / A2, a = r - ts * A2;
      unsigned* dst = reinterpret_cast<unsigned*>(Hs + ci * t.hld + r * d.B);
      const int tt = (t0 - 1 + ts + d.T) % d.T;
      const unsigned* src = ci < Cin
          ? reinterpret_cast<const unsigned*>(h + ((long long)s * Cin + ci) * S + tt * AB +
                                              wrap1(a - 1, d.A) * d.B)
          : nullptr;
      const int nw = d.B / 2;
      unsigned prev = src ? src[nw - 1] : 0u, cur = src ? src[0] : 0u;
      for (int i = 0; i < nw; ++i) {
        const unsigned next = src ? src[i + 1 < nw ? i + 1 : 0] : 0u;
        dst[i] = __byte_perm(prev, cur, 0x5432);              // h[b - 1], h[b]
        dst[copy / 2 + i] = cur;                              // h[b], h[b + 1]
        dst[copy + i] = __byte_perm(cur, next, 0x5432);       // h[b + 1], h[b + 2]
        prev = cur;
        cur = next;
      }
    }
    for (int e = tid; e < 3 * NC * 8 * ((t.hld - rows * d.B) / 2); e += kBwThreads) {
      const int pad = (t.hld - rows * d.B) / 2, c = e / pad;   // read by the padded positions
      reinterpret_cast<unsigned*>(Hs + c * t.hld + rows * d.B)[e - c * pad] = 0u;
    }
    __syncthreads();
    float acc[MT][3][NC][4], ab[MT][4];
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        ab[m][i] = 0.f;
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int c = 0; c < NC; ++c) acc[m][b][c][i] = 0.f;
      }
    const unsigned ga = (unsigned)__cvta_generic_to_shared(Gs) +
                        ((lane & 15) * t.gld + (lane >> 4) * 8) * 2;
    for (int ts = 0; ts < t.TT; ++ts) {
      const __nv_bfloat16* hb = Hs + (lane >> 2) * t.hld + ((ts + 1 + dt) * A2 + 1 + da) * d.B +
                                2 * (lane & 3);
      auto positions = [&](int q, auto steps) {   // 16 positions each
        constexpr int K = decltype(steps)::value;
        unsigned af[MT][K][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
          for (int k = 0; k < K; ++k)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                         : "=r"(af[m][k][0]), "=r"(af[m][k][1]), "=r"(af[m][k][2]), "=r"(af[m][k][3])
                         : "r"(ga + (m * 16 * t.gld + ts * t.ABp + q + 16 * k) * 2));
#pragma unroll
        for (int b = 0; b < 3; ++b)
#pragma unroll
          for (int c = 0; c < NC; ++c) {
            const unsigned* hw = reinterpret_cast<const unsigned*>(hb + b * copy + c * 8 * t.hld + q);
            unsigned bf[K][2];
#pragma unroll
            for (int k = 0; k < K; ++k) bf[k][0] = hw[8 * k], bf[k][1] = hw[8 * k + 4];
#pragma unroll
            for (int m = 0; m < MT; ++m) add_products<K>(acc[m][b][c], af[m], bf);
          }
        if (warp == 4) {   // a column of ones: the bias gradient
          unsigned ones[K][2];
#pragma unroll
          for (int k = 0; k < K; ++k) ones[k][0] = ones[k][1] = 0x3f803f80u;
#pragma unroll
          for (int m = 0; m < MT; ++m) add_products<K>(ab[m], af[m], ones);
        }
      };
      int q = 0;
      for (; q + 32 <= t.ABp; q += 32) positions(q, std::integral_constant<int, 2>());
      if (q < t.ABp) positions(q, std::integral_constant<int, 1>());
    }
#pragma unroll
    for (int m = 0; m < MT; ++m) {
#pragma unroll
      for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < NC; ++c)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            float& v = sums[(((m * 3 + b) * NC + c) * 4 + i) * kBwThreads + tid];
            v = __fadd_rn(v, acc[m][b][c][i]);
          }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float& v = sums[(MT * 3 * NC * 4 + m * 4 + i) * kBwThreads + tid];
        v = __fadd_rn(v, ab[m][i]);
      }
    }
  }
  // this CTA's sums in the layout of the gradient: weights, then biases
  float* out = part + (long long)blockIdx.x * P;
  for (int m = 0; m < MT; ++m)
    for (int i = 0; i < 4; ++i) {
      const int co = m * 16 + (lane >> 2) + (i >> 1) * 8;
      if (co >= Cout) continue;
      for (int b = 0; b < 3; ++b)
        for (int c = 0; c < NC; ++c) {
          const int ci = c * 8 + 2 * (lane & 3) + (i & 1);
          if (ci < Cin)
            out[((long long)co * Cin + ci) * kK + warp * 3 + b] =
                sums[(((m * 3 + b) * NC + c) * 4 + i) * kBwThreads + tid];
        }
      if (warp == 4 && (lane & 3) == 0 && (i & 1) == 0)
        out[(long long)Cout * Cin * kK + co] = sums[(MT * 3 * NC * 4 + m * 4 + i) * kBwThreads + tid];
    }
}

__global__ void k_cg_sum(const float* __restrict__ part, int P, int parts, float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P) return;
  float s = 0.f, low = 0.f;   // (with what each addition rounds off, by TwoSum)
#pragma unroll 8
  for (int c = 0; c < parts; ++c) {
    const float x = part[(long long)c * P + i], t = __fadd_rn(s, x), z = __fsub_rn(t, s);
    low = __fadd_rn(low, __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z)));
    s = t;
  }
  out[i] = __fadd_rn(s, low);
}

__global__ void k_cg_adam(float* __restrict__ th, const float* __restrict__ gr,
                          float* __restrict__ m, float* __restrict__ v, long long n, float lr,
                          float c1, float c2, __nv_bfloat16* __restrict__ thb) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x) {
    const float gi = gr[i];
    const float mi = 0.9f * m[i] + 0.1f * gi;
    const float vi = 0.999f * v[i] + 0.001f * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float x = th[i] - lr * (mi / c1) / (sqrtf(vi / c2) + 1e-8f);
    th[i] = x;
    thb[i] = __float2bfloat16_rn(x);
  }
}

__global__ void k_cg_to_bf16(const float* __restrict__ x, long long n, __nv_bfloat16* __restrict__ y) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n;
       i += (long long)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16_rn(x[i]);
}

__global__ void k_cg_noise(long long n0, int n, int S, uint32_t stream, uint32_t k0, uint32_t k1,
                           __nv_bfloat16* __restrict__ z) {
  const long long total = (long long)n * S;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(e / S), p = (int)(e - (long long)s * S);
    uint32_t c[4] = {(uint32_t)p, (uint32_t)(n0 + s), stream, kTagNoise};
    philox4x32_10(c, k0, k1);
    const float u1 = (float)(((double)c[0] + 0.5) * 2.3283064365386962890625e-10);
    const float u2 = (float)((double)c[1] * 2.3283064365386962890625e-10);
    const float r = sqrtf(-2.f * logf(u1));
    z[e] = __float2bfloat16_rn(r * cosf(6.283185307179586f * u2));
  }
}

__global__ void k_cg_draw(const float* __restrict__ logits, long long n0, int n, int S,
                          uint32_t stream, uint32_t k0, uint32_t k1, int8_t* __restrict__ f) {
  const long long total = (long long)n * S;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(e / S), p = (int)(e - (long long)s * S);
    uint32_t c[4] = {(uint32_t)p, (uint32_t)(n0 + s), stream, kTagDraw};
    philox4x32_10(c, k0, k1);
    const double u = (double)c[0] * 2.3283064365386962890625e-10;
    const double pr = 1.0 / (1.0 + exp(-(double)logits[e]));
    f[e] = u < pr ? (int8_t)1 : (int8_t)-1;
  }
}

int grid_for(long long n, int threads) {
  const long long b = (n + threads - 1) / threads;
  return (int)(b < 4096 ? (b > 0 ? b : 1) : 4096);
}

}  // namespace

struct nmc_cgen {
  Dims d{};
  int C = 0, max_batch = 0;
  uint64_t seed = 0;
  cudaStream_t st = nullptr;
  int device = 0;
  int cin[kLayers], cout[kLayers];
  long long oW[kLayers], ob[kLayers], P = 0;
  float *th = nullptr, *gr = nullptr, *m = nullptr, *v = nullptr, *logits = nullptr;
  __nv_bfloat16 *thb = nullptr, *act[kLayers] = {}, *gA = nullptr, *gB = nullptr;
  double* dloss = nullptr;
  // the weights as k_cg_conv reads them (FP32, per layer forward and backward), and the
  // partial sums of k_cg_bwd_w_tc ([parts][the largest layer]), where the largest call takes those kernels
  float *wf[kLayers] = {}, *wb[kLayers] = {}, *part = nullptr;
  int parts = 0;
  long long steps = 0;
  std::vector<void*> allocs;
};

namespace {

template <typename T>
nmc_status cg_alloc(nmc_cgen* g, T*& p, long long n) {
  if (cudaMalloc((void**)&p, (size_t)(n > 0 ? n : 1) * sizeof(T)) != cudaSuccess) {
    cudaGetLastError();
    p = nullptr;
    return NMC_ENOMEM;
  }
  g->allocs.push_back(p);
  return NMC_OK;
}

#define CG_TRY(expr)                  \
  do {                                \
    const nmc_status s_ = (expr);     \
    if (s_ != NMC_OK) return s_;      \
  } while (0)

nmc_status cg_last(void) {
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? NMC_OK : NMC_ECUDA;
}

constexpr size_t kConvSmem = 200 * 1024;

// Shared memory of a k_cg_conv tile of PT positions and cos channels: the slices that PT
// consecutive positions touch at most, and their halo
size_t conv_smem(const Dims& d, int Cin, int PT, int cos) {
  const int AB = d.A * d.B;
  int ns = PT % AB == 0 ? PT / AB : AB % PT == 0 ? 1 : (PT - 2) / AB + 2;
  if (ns > d.T) ns = d.T;
  const size_t words = (size_t)((Cin + 1) / 2) * (ns + 2) * (d.A + 2) * (d.B + 2);
  return ((words + 3) & ~(size_t)3) * 4 + 2 * 3 * (size_t)Cin * cos * 4;
}

// From how many outputs of a middle layer on the tiled kernel takes the convolutions: it keeps 16 to 64
// sums per thread and one or two CTAs per SM, so below, most of the GPU waits for a few, and one output
// per thread is faster. us a sampling call, one per thread / tiled (outputs): 8 channels 61 / 81 (15 k),
// 88 / 84 (95 k), 115 / 84 (192 k); 16 channels 72 / 101 (10 k), 113 / 106 (123 k), 166 / 106 (246 k);
// 32 channels 90 / 150 (20 k), 149 / 152 (123 k), 234 / 156 (246 k). The bits are the same.
constexpr long long kTileOutputs = 125000;
// The same for the weight gradients, in positions: the one product has a fixed cost of some 25 us (8
// channels) to 60 (32) a call. us a gradient call, a CTA per channel pair / one product (positions): 8
// channels 138 / 159 (1280), 171 / 166 (2560), 242 / 194 (6000); 16 channels 165 / 196 (1280), 208 / 211
// (2560), 313 / 268 (6000); 32 channels 231 / 272 (960), 369 / 344 (2560), 505 / 409 (4000).
constexpr long long kTcPositions = 2600;

// One convolution (or its transpose) by the tiled kernel; false: its halo does not fit or there are too
// few outputs. 256
// positions per CTA, or 64 while those would not give every SM two CTAs (37 x 1080 positions, 32
// channels: 121 us per middle layer with 64, 127 with 128).
template <int MODE>
bool conv_tiled(nmc_cgen* g, const __nv_bfloat16* in, int Cin, const float* wt, const float* bias,
                int Cout, int n, const __nv_bfloat16* act, __nv_bfloat16* out_h, float* out_f) {
  const int S = g->d.S();
  if ((long long)n * S * g->C < kTileOutputs) return false;
  auto run = [&](auto kernel, int TP, int TC) {
    const int groups = (Cout + TC - 1) / TC, wco = TC == 2 ? 1 : groups >= 3 ? 4 : groups;
    const int PT = kConvThreads / wco * TP;
    const size_t bytes = conv_smem(g->d, Cin, PT, TC * wco);
    if (bytes > kConvSmem) return false;
    const dim3 grid((S + PT - 1) / PT, (groups + wco - 1) / wco, n);
    if (TP > 2 && (long long)grid.x * grid.y * grid.z < 2 * nmc::sm_count()) return false;
    nmc::allow_max_dynamic_smem((const void*)kernel);
    kernel<<<grid, kConvThreads, bytes, g->st>>>(in, Cin, wt, pad8(Cout), bias, Cout, g->d, wco,
                                                 act, out_h, out_f);
    return true;
  };
  if (Cout <= 2) return run(k_cg_conv<2, 2, MODE>, 2, 2);
  return run(k_cg_conv<8, 8, MODE>, 8, 8) || run(k_cg_conv<2, 8, MODE>, 2, 8);
}

void forward(nmc_cgen* g, int n) {
  const int S = g->d.S();
  for (int j = 0; j < kLayers; ++j) {
    const bool last = j == kLayers - 1;
    __nv_bfloat16* oh = last ? nullptr : g->act[j + 1];
    float* of = last ? g->logits : nullptr;
    if (last ? conv_tiled<kLogits>(g, g->act[j], g->cin[j], g->wf[j], g->th + g->ob[j], g->cout[j],
                                   n, nullptr, oh, of)
             : conv_tiled<kHidden>(g, g->act[j], g->cin[j], g->wf[j], g->th + g->ob[j], g->cout[j],
                                   n, nullptr, oh, of))
      continue;
    const dim3 grid((S + kFwdThreads - 1) / kFwdThreads, g->cout[j], n);
    k_cg_fwd<<<grid, kFwdThreads, g->cin[j] * kK * sizeof(float), g->st>>>(
        g->act[j], g->cin[j], g->thb + g->oW[j], g->th + g->ob[j], g->cout[j], g->d, last ? 0 : 1,
        oh, of);
  }
}

// Weight and bias gradients of one layer as one product over all positions; false: rows of odd
// length (a pair of positions would straddle two), more than 32 channels, too few positions, or
// slices that do not fit shared memory.
bool bwd_w_tc(nmc_cgen* g, int j, const __nv_bfloat16* gin, int n) {
  const Dims& d = g->d;
  const int Cin = g->cin[j], Cout = g->cout[j];
  if ((long long)n * d.S() < kTcPositions) return false;
  if (d.B % 2 || Cin > 32 || Cout > 32 || !g->part) return false;
  const int MT = Cout > 16 ? 2 : 1, NC = Cin > 16 ? 4 : Cin > 8 ? 2 : 1;
  BwTile t{};
  t.ABp = (d.A * d.B + 15) & ~15;
  size_t bytes = 0;
  for (t.TT = d.T < 8 ? d.T : 8; t.TT > 0; --t.TT) {
    t.gld = t.TT * t.ABp + 8;
    t.hld = (t.TT + 2) * (d.A + 2) * d.B + 16;
    t.hld += (72 - t.hld % 64) % 64;   // 8 mod 64: eight channels' words on different banks
    bytes = (size_t)(MT * 3 * NC * 4 + MT * 4) * kBwThreads * 4 +
            2 * ((size_t)MT * 16 * t.gld + (size_t)3 * NC * 8 * t.hld);
    if (bytes <= 226 * 1024) break;
  }
  if (t.TT == 0) return false;
  t.per_sample = (d.T + t.TT - 1) / t.TT;
  t.total = n * t.per_sample;
  const int P = Cout * Cin * kK + Cout, parts = t.total < g->parts ? t.total : g->parts;
  auto run = [&](auto kernel) {
    nmc::allow_max_dynamic_smem((const void*)kernel);
    kernel<<<parts, kBwThreads, bytes, g->st>>>(gin, Cout, g->act[j], Cin, d, t, g->part, P);
  };
  if (MT == 2) NC == 4 ? run(k_cg_bwd_w_tc<2, 4>) : NC == 2 ? run(k_cg_bwd_w_tc<2, 2>) : run(k_cg_bwd_w_tc<2, 1>);
  else NC == 4 ? run(k_cg_bwd_w_tc<1, 4>) : NC == 2 ? run(k_cg_bwd_w_tc<1, 2>) : run(k_cg_bwd_w_tc<1, 1>);
  k_cg_sum<<<(P + 127) / 128, 128, 0, g->st>>>(g->part, P, parts, g->gr + g->oW[j]);
  return true;
}

// loss of the current logits against d_fields into g->dloss (sum), gradients into g->gr
void backward(nmc_cgen* g, const int8_t* d_fields, int n) {
  const int S = g->d.S();
  const long long total = (long long)n * S;
  cudaMemsetAsync(g->dloss, 0, sizeof(double), g->st);
  k_cg_loss<<<grid_for(total, kWThreads), kWThreads, 0, g->st>>>(
      g->logits, d_fields, total, 1.f / (float)total, g->gA, g->dloss);
  __nv_bfloat16* gcur = g->gA;
  __nv_bfloat16* gnext = g->gB;
  for (int j = kLayers - 1; j >= 0; --j) {
    if (!bwd_w_tc(g, j, gcur, n))
      k_cg_bwd_w<<<dim3(g->cin[j], g->cout[j]), kWThreads, 0, g->st>>>(
          gcur, g->cout[j], g->act[j], g->cin[j], g->d, n, g->gr + g->oW[j], g->gr + g->ob[j]);
    if (j > 0) {
      if (!conv_tiled<kBackward>(g, gcur, g->cout[j], g->wb[j], nullptr, g->cin[j], n, g->act[j],
                                 gnext, nullptr)) {
        const dim3 grid((S + kFwdThreads - 1) / kFwdThreads, g->cin[j], n);
        k_cg_bwd_in<<<grid, kFwdThreads, g->cout[j] * kK * sizeof(float), g->st>>>(
            gcur, g->cout[j], g->thb + g->oW[j], g->cin[j], g->d, g->act[j], gnext);
      }
      __nv_bfloat16* t = gcur;
      gcur = gnext;
      gnext = t;
    }
  }
}

// the convolutions' layouts of the current BF16 weights, if any call reads them (a launch of some 5 us
// behind every change of the weights)
void layout(nmc_cgen* g) {
  if (!g->wf[0]) return;
  LayoutArgs a;
  int most = 0;
  for (int j = 0; j < kLayers; ++j) {
    const int ci = g->cin[j], co = g->cout[j];
    a.W[j] = g->thb + g->oW[j];
    a.wf[j] = g->wf[j];
    a.wb[j] = g->wb[j];
    a.cin[j] = ci;
    a.cout[j] = co;
    most = std::max(most, kK * (ci * pad8(co) + co * pad8(ci)));
  }
  k_cg_layout<<<dim3(grid_for(most, 256), kLayers), 256, 0, g->st>>>(a);
}

void noise(nmc_cgen* g, long long n0, int n, uint32_t stream) {
  const int S = g->d.S();
  k_cg_noise<<<grid_for((long long)n * S, 256), 256, 0, g->st>>>(
      n0, n, S, stream, (uint32_t)g->seed, (uint32_t)(g->seed >> 32), g->act[0]);
}

}  // namespace

extern "C" {

nmc_status nmc_cgen_create(int Lx, int Ly, int L_tau, int channels, uint64_t seed, int max_batch,
                           void* cuda_stream, nmc_cgen** out) {
  if (!out) return NMC_EINVAL;
  *out = nullptr;
  if (Lx < 1 || Ly < 1 || L_tau < 1 || channels < 1 || channels > 64 || max_batch < 1 ||
      (long long)Lx * Ly * L_tau > (1 << 24) || max_batch > 65535)
    return NMC_EINVAL;
  nmc_cgen* g = new (std::nothrow) nmc_cgen();
  if (!g) return NMC_ENOMEM;
  g->d = Dims{L_tau, Ly, Lx};
  g->C = channels;
  g->max_batch = max_batch;
  g->seed = seed;
  g->st = (cudaStream_t)cuda_stream;
  cudaGetDevice(&g->device);
  const int C = channels;
  const int ci[kLayers] = {1, C, C, C}, co[kLayers] = {C, C, C, 1};
  long long off = 0;
  for (int j = 0; j < kLayers; ++j) {
    g->cin[j] = ci[j];
    g->cout[j] = co[j];
    g->oW[j] = off;
    off += (long long)co[j] * ci[j] * kK;
    g->ob[j] = off;
    off += co[j];
  }
  g->P = off;
  const long long S = g->d.S(), nb = max_batch;
  nmc_status s = NMC_OK;
  if (s == NMC_OK) s = cg_alloc(g, g->th, g->P);
  if (s == NMC_OK) s = cg_alloc(g, g->gr, g->P);
  if (s == NMC_OK) s = cg_alloc(g, g->m, g->P);
  if (s == NMC_OK) s = cg_alloc(g, g->v, g->P);
  if (s == NMC_OK) s = cg_alloc(g, g->thb, g->P);
  if (s == NMC_OK) s = cg_alloc(g, g->logits, nb * S);
  for (int j = 0; j < kLayers && s == NMC_OK; ++j) s = cg_alloc(g, g->act[j], nb * ci[j] * S);
  if (s == NMC_OK) s = cg_alloc(g, g->gA, nb * C * S);
  if (s == NMC_OK) s = cg_alloc(g, g->gB, nb * C * S);
  if (s == NMC_OK) s = cg_alloc(g, g->dloss, 1);
  for (int j = 0; j < kLayers && nb * S * C >= kTileOutputs; ++j) {
    if (s == NMC_OK) s = cg_alloc(g, g->wf[j], (long long)kK * ci[j] * pad8(co[j]));
    if (s == NMC_OK) s = cg_alloc(g, g->wb[j], (long long)kK * co[j] * pad8(ci[j]));
  }
  if (Lx % 2 == 0 && C <= 32 && nb * S >= kTcPositions) {
    g->parts = nmc::sm_count();
    if (s == NMC_OK) s = cg_alloc(g, g->part, g->parts * ((long long)C * C * kK + C));
  }
  if (s != NMC_OK) {
    nmc_cgen_destroy(g);
    return s;
  }
  // Glorot-uniform weights, zero biases
  std::vector<float> th((size_t)g->P, 0.f);
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  for (int j = 0; j < kLayers; ++j) {
    const double bound = std::sqrt(6.0 / (kK * (double)(ci[j] + co[j])));
    for (long long e = 0; e < (long long)co[j] * ci[j] * kK; ++e) {
      uint32_t c[4] = {(uint32_t)e, (uint32_t)j, 0u, kTagInit};
      philox4x32_10(c, k0, k1);
      const double u = (double)c[0] * 2.3283064365386962890625e-10;
      th[(size_t)(g->oW[j] + e)] = (float)((2.0 * u - 1.0) * bound);
    }
  }
  s = nmc_cgen_set_params(g, th.data());
  if (s != NMC_OK) {
    nmc_cgen_destroy(g);
    return s;
  }
  *out = g;
  return NMC_OK;
}

nmc_status nmc_cgen_n_params(const nmc_cgen* g, long long* n) {
  if (!g || !n) return NMC_EINVAL;
  *n = g->P;
  return NMC_OK;
}

nmc_status nmc_cgen_get_params(const nmc_cgen* g, float* theta) {
  if (!g || !theta) return NMC_EINVAL;
  if (cudaMemcpyAsync(theta, g->th, (size_t)g->P * sizeof(float), cudaMemcpyDeviceToHost, g->st) !=
          cudaSuccess ||
      cudaStreamSynchronize(g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  return NMC_OK;
}

nmc_status nmc_cgen_set_params(nmc_cgen* g, const float* theta) {
  if (!g || !theta) return NMC_EINVAL;
  const size_t b = (size_t)g->P * sizeof(float);
  if (cudaMemcpyAsync(g->th, theta, b, cudaMemcpyHostToDevice, g->st) != cudaSuccess ||
      cudaMemsetAsync(g->m, 0, b, g->st) != cudaSuccess ||
      cudaMemsetAsync(g->v, 0, b, g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  k_cg_to_bf16<<<grid_for(g->P, 256), 256, 0, g->st>>>(g->th, g->P, g->thb);
  layout(g);
  g->steps = 0;
  if (cudaStreamSynchronize(g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  return cg_last();
}

nmc_status nmc_cgen_forward(nmc_cgen* g, const float* d_z, int n, float* d_logits) {
  if (!g || !d_z || !d_logits || n < 1 || n > g->max_batch) return NMC_EINVAL;
  const long long total = (long long)n * g->d.S();
  k_cg_to_bf16<<<grid_for(total, 256), 256, 0, g->st>>>(d_z, total, g->act[0]);
  forward(g, n);
  if (cudaMemcpyAsync(d_logits, g->logits, (size_t)total * sizeof(float),
                      cudaMemcpyDeviceToDevice, g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  return cg_last();
}

nmc_status nmc_cgen_loss_grad(nmc_cgen* g, const float* d_z, const int8_t* d_fields, int n,
                              double* loss, float* d_grad) {
  if (!g || !d_z || !d_fields || !loss || !d_grad || n < 1 || n > g->max_batch) return NMC_EINVAL;
  const long long total = (long long)n * g->d.S();
  k_cg_to_bf16<<<grid_for(total, 256), 256, 0, g->st>>>(d_z, total, g->act[0]);
  forward(g, n);
  backward(g, d_fields, n);
  double sum = 0.0;
  if (cudaMemcpyAsync(d_grad, g->gr, (size_t)g->P * sizeof(float), cudaMemcpyDeviceToDevice,
                      g->st) != cudaSuccess ||
      cudaMemcpyAsync(&sum, g->dloss, sizeof(double), cudaMemcpyDeviceToHost, g->st) != cudaSuccess ||
      cudaStreamSynchronize(g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  *loss = sum / (double)total;
  return cg_last();
}

nmc_status nmc_cgen_train_step(nmc_cgen* g, const int8_t* d_fields, int n, long long sample0,
                               float lr, double* loss) {
  if (!g || !d_fields || n < 1 || n > g->max_batch || sample0 < 0) return NMC_EINVAL;
  noise(g, sample0, n, 0u);
  forward(g, n);
  backward(g, d_fields, n);
  ++g->steps;
  const float c1 = 1.f - std::pow(0.9f, (float)g->steps);
  const float c2 = 1.f - std::pow(0.999f, (float)g->steps);
  k_cg_adam<<<grid_for(g->P, 256), 256, 0, g->st>>>(g->th, g->gr, g->m, g->v, g->P, lr, c1, c2,
                                                    g->thb);
  layout(g);
  if (loss) {
    double sum = 0.0;
    if (cudaMemcpyAsync(&sum, g->dloss, sizeof(double), cudaMemcpyDeviceToHost, g->st) !=
            cudaSuccess ||
        cudaStreamSynchronize(g->st) != cudaSuccess) {
      cudaGetLastError();
      return NMC_ECUDA;
    }
    *loss = sum / ((double)n * g->d.S());
  }
  return cg_last();
}

nmc_status nmc_cgen_sample(nmc_cgen* g, long long n0, int n, int8_t* d_fields, float* d_logits) {
  if (!g || !d_fields || n < 1 || n > g->max_batch || n0 < 0) return NMC_EINVAL;
  const int S = g->d.S();
  noise(g, n0, n, 1u);
  forward(g, n);
  k_cg_draw<<<grid_for((long long)n * S, 256), 256, 0, g->st>>>(
      g->logits, n0, n, S, 1u, (uint32_t)g->seed, (uint32_t)(g->seed >> 32), d_fields);
  if (d_logits &&
      cudaMemcpyAsync(d_logits, g->logits, (size_t)n * S * sizeof(float), cudaMemcpyDeviceToDevice,
                      g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  if (cudaStreamSynchronize(g->st) != cudaSuccess) {
    cudaGetLastError();
    return NMC_ECUDA;
  }
  return cg_last();
}

void nmc_cgen_destroy(nmc_cgen* g) {
  if (!g) return;
  if (g->st) cudaStreamSynchronize(g->st);
  else cudaDeviceSynchronize();
  for (void* p : g->allocs) cudaFree(p);
  cudaGetLastError();
  delete g;
}

}  // extern "C"
