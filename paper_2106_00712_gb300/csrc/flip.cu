// Local Metropolis updates of one time slice with rank-k delayed Green's function updates.
//
// One CTA per chain handles both spins. For slice l the CTA draws the N Philox uniforms
// u_i (counter (l*N+i, sweep, chain, 0)), then visits i = 0..N-1 in order:
//   G^_ii = G0_ii + sum_{q<m} a_q[i] b_q[i]                    (warp 0, both spins)
//   R^sigma = 1 + Delta^sigma (1 - G^_ii), Delta^sigma = e^{-2 sigma lam s} - 1 (FP64)
//   accept iff u_i < |R^up R^dn|
// and on acceptance appends the Sherman-Morrison vectors of the flip,
//   a_m = -(Delta/R^sigma) (e_i - G^_{:,i}),   b_m = G^_{i,:},
// each computed from G0 and the m earlier pairs (all threads). When m reaches k, or at
// the end of the slice, the k pairs are folded into G0 as one rank-k update
// G0 += A B^T. In exact arithmetic this equals applying each rank-1 update at once.
// G0 of both spins sits in shared memory when it fits (N <= 64 in FP64), else in global
// memory (L2); the panels always live in shared memory (k is clamped to fit).
// That is k_flip in FP32, and in FP64 for small k and above some 560 sites; and k_flip_df in FP32 pairs
// for small k, and without tensor cores for most sizes. Elsewhere FP64 and FP32 pairs take k_flip_block,
// which decides blocks of up to min(k, 16) sites apart (the rules stand at flip_slice).
#include <cooperative_groups.h>

#include "fold16.cuh"
#include "nmc_internal.cuh"
#include "quotient.cuh"

namespace cg = cooperative_groups;

namespace nmc {

namespace {

NMC_DEBUG_FLAG

constexpr int kThreads = 256;
// compensated kernel: 256 threads for the panel entries (one entry of G^'s column or row each
// at N = 64) plus one warp whose first thread evaluates the ratio meanwhile
constexpr int kPanelThreads = 256;
constexpr int kThreadsDf = kPanelThreads + 32;

// Thread t owns column c = t % N of rows t / N, t / N + rows_per_pass, ... of both spins:
// 32-bit index arithmetic only, consecutive threads on consecutive columns.
template <typename T>
__device__ void flush(T* G, const T* Ap, const T* Bp, int m, int N, int KK, long long NN,
                      int ns) {
  // G[sp][r][c] += sum_{q<m} A[sp][q][r] * B[sp][q][c]
  const int nthr = blockDim.x;
  if ((int)threadIdx.x >= (nthr / N) * N && nthr >= N) return;
  const int c0 = threadIdx.x % N, r0 = threadIdx.x / N;
  const int rstep = nthr >= N ? nthr / N : 1;
  for (int sp = 0; sp < ns; ++sp) {
    const T* A_ = Ap + sp * KK * N;
    const T* B_ = Bp + sp * KK * N;
    T* Gs = G + sp * NN;
    for (int c = c0; c < N; c += (nthr >= N ? N : nthr)) {
      for (int r = (nthr >= N ? r0 : 0); r < N; r += rstep) {
        T v = Gs[r * N + c];
        for (int q = 0; q < m; ++q) v = fma(A_[q * N + r], B_[q * N + c], v);
        Gs[r * N + c] = v;
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kThreads, 2) k_flip(const FlipArgs<T> f) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_accept[2];  // by attempt parity: see the loop
  __shared__ double s_coef[2];
  __shared__ double s_sign;
  __shared__ unsigned long long s_cnt[3];

  const int c = blockIdx.x;
  const int N = f.N, KK = f.kk;
  const long long NN = (long long)N * N;
  const int ns = f.ns;
  T* Ap = (T*)smraw;                // [ns][KK][N]
  T* Bp = Ap + ns * KK * N;         // [ns][KK][N]
  T* diag = Bp + ns * KK * N;       // [ns][N]
  T* Gs = diag + ns * N;            // [ns][N][N] when g_in_smem
  double* u = (double*)(((uintptr_t)(Gs + (f.g_in_smem ? ns * NN : 0)) + 15) & ~(uintptr_t)15);
  int8_t* sl = (int8_t*)(u + N);

  T* Gg = f.G + (long long)c * ns * NN;
  T* G = f.g_in_smem ? Gs : Gg;
  int8_t* fl = f.fields + ((long long)c * f.L + f.l) * N;
  // Philox counter words of this chain: its global index, and sweeps since its start
  const uint32_t gchain = (uint32_t)(f.chain_id ? f.chain_id[c] : f.chain_offset + c);
  const uint32_t sweep = (uint32_t)((f.ctr ? f.ctr[0] : (long long)f.sweep) -
                                    (f.sweep_base ? f.sweep_base[c] : 0));
  const uint8_t* rp = f.replay ? f.replay + ((long long)c * f.L + f.l) * N : nullptr;

  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    sl[i] = fl[i];
    uint32_t ctr[4] = {(uint32_t)(f.l * N + i), sweep, gchain, kTagFlip};
    philox4x32_10(ctr, f.key0, f.key1);
    u[i] = (double)ctr[0] * 2.3283064365386962890625e-10;  // 2^-32
  }
  if (f.g_in_smem)
    for (long long e = threadIdx.x; e < ns * NN; e += blockDim.x) Gs[e] = Gg[e];
  if (threadIdx.x == 0) {
    s_sign = f.sign[c];
    s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ns * N; i += blockDim.x) {
    const int sp = i / N, r = i % N;
    diag[i] = G[sp * NN + (long long)r * N + r];
  }
  __syncthreads();

  // The accept flag is double-buffered by attempt parity: after a rejection there is one
  // barrier per attempt, so thread 0 may write the next attempt's flag while slower threads
  // still read this one. It cannot write this slot again (attempt i+2) before every thread
  // has passed attempt i+1's barrier, which follows its read of attempt i's flag.
  int m = 0;
  for (int i = 0; i < N; ++i) {
    if (threadIdx.x < 32) {
      const int lane = threadIdx.x, sp = lane >> 4, q0 = lane & 15;
      const T* A_ = Ap + sp * KK * N;
      const T* B_ = Bp + sp * KK * N;
      T sum = T(0);
      if (sp < ns)
        for (int q = q0; q < m; q += 16) sum = fma(A_[q * N + i], B_[q * N + i], sum);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const T sum_dn = __shfl_sync(0xffffffffu, sum, 16);
      if (lane == 0) {
        const double gu = (double)(diag[i] + sum);
        const int s = sl[i];
        const double du = (s > 0) ? f.dm : f.dp;  // e^{-2 lam s} - 1
        const double dd = (s > 0) ? f.dp : f.dm;  // e^{+2 lam s} - 1
        const double Ru = 1.0 + du * (1.0 - gu);
        // spin down: 1 - G^dn_ii, or G^up_ii when G_dn = I - P G_up^T P
        const double Rd = 1.0 + dd * (ns == 2 ? 1.0 - (double)(diag[N + i] + sum_dn) : gu);
        const double R = Ru * Rd;
        const bool mine = u[i] < fabs(R);
        bool acc = mine;
        if (rp) {
          acc = rp[i] != 0;
          if (acc != mine) s_cnt[2]++;
        }
        s_cnt[0]++;
        s_accept[i & 1] = acc ? 1 : 0;
        if (acc) {
          s_coef[0] = -du / Ru;
          s_coef[1] = -dd / Rd;
          if (R < 0.0) s_sign = -s_sign;
          s_cnt[1]++;
          sl[i] = (int8_t)(-s);
        }
      }
    }
    __syncthreads();
    if (s_accept[i & 1]) {
      const T coef0 = (T)s_coef[0], coef1 = (T)s_coef[1];
      for (int t = threadIdx.x; t < 2 * ns * N; t += blockDim.x) {
        const int sp = t / (2 * N);
        const int kind = (t / N) & 1;
        const int r = t % N;
        const T* Gsp = G + sp * NN;
        const T* A_ = Ap + sp * KK * N;
        const T* B_ = Bp + sp * KK * N;
        if (kind == 0) {  // column i of G^: a_m = coef (e_i - G^_{:,i})
          T v = Gsp[(long long)r * N + i];
          for (int q = 0; q < m; ++q) v = fma(A_[q * N + r], B_[q * N + i], v);
          if (NMC_DCHECK(m < KK && sp < ns && r < N, 111))
            Ap[(sp * KK + m) * N + r] = (sp ? coef1 : coef0) * ((r == i ? T(1) : T(0)) - v);
        } else {          // row i of G^: b_m = G^_{i,:}
          T v = Gsp[(long long)i * N + r];
          for (int q = 0; q < m; ++q) v = fma(A_[q * N + i], B_[q * N + r], v);
          if (NMC_DCHECK(m < KK && sp < ns && r < N, 112)) Bp[(sp * KK + m) * N + r] = v;
        }
      }
      ++m;
      __syncthreads();
      if (m == KK) {
        flush(G, Ap, Bp, m, N, KK, NN, f.ns);
        m = 0;
        __syncthreads();
        for (int j = threadIdx.x; j < ns * N; j += blockDim.x) {
          const int sp = j / N, r = j % N;
          diag[j] = G[sp * NN + (long long)r * N + r];
        }
        __syncthreads();
      }
    }
  }
  if (m > 0) {
    flush(G, Ap, Bp, m, N, KK, NN, f.ns);
    __syncthreads();
  }
  if (f.g_in_smem)
    for (long long e = threadIdx.x; e < ns * NN; e += blockDim.x) Gg[e] = Gs[e];
  for (int i = threadIdx.x; i < N; i += blockDim.x) fl[i] = sl[i];
  if (threadIdx.x == 0) {
    f.sign[c] = s_sign;
    f.counts[3 * c + 0] += s_cnt[0];
    f.counts[3 * c + 1] += s_cnt[1];
    f.counts[3 * c + 2] += s_cnt[2];
  }
}

// Double-float variant. G0, the rank-k panels and every multiply-add are FP32 pairs
// (df.cuh), and a running diagonal dg_j = G^_jj is updated with each accepted flip
// (dg_j += a_m[j] b_m[j]), so an attempt reads G^_ii directly instead of reducing over
// the panels. The acceptance is the FP64 decision u < |R|: R is first evaluated in
// double-float (relative error ~1e-13); when |u - |R|| exceeds a margin of 1e-10 (|R| + 1)
// that value decides, and only inside the margin is R recomputed in FP64 from the same
// G^_ii -- both give the FP64 decision. The update coefficient -Delta/R^sigma uses a
// double-float reciprocal.
__device__ void flush_df(df2* G, const df2* Ap, const df2* Bp, int m, int N, int KK,
                         long long NN, int ns) {
  const int nthr = blockDim.x;
  if ((int)threadIdx.x >= (nthr / N) * N && nthr >= N) return;
  const int c0 = threadIdx.x % N, r0 = threadIdx.x / N;
  const int rstep = nthr >= N ? nthr / N : 1;
  for (int sp = 0; sp < ns; ++sp) {
    const df2* A_ = Ap + sp * KK * N;
    const df2* B_ = Bp + sp * KK * N;
    df2* Gs = G + sp * NN;
    for (int c = c0; c < N; c += (nthr >= N ? N : nthr)) {
      int r = nthr >= N ? r0 : 0;
      // four rows at a time: four independent accumulation chains share each B load
      // (every output still sees the same operations in the same order)
      for (; r + 3 * rstep < N; r += 4 * rstep) {
        df2 a0 = Gs[r * N + c], a1 = Gs[(r + rstep) * N + c];
        df2 a2 = Gs[(r + 2 * rstep) * N + c], a3 = Gs[(r + 3 * rstep) * N + c];
        for (int q = 0; q < m; ++q) {
          const df2 bq = B_[q * N + c];
          const df2* Aq = A_ + q * N + r;
          df_fma_acc(a0, Aq[0], bq);
          df_fma_acc(a1, Aq[rstep], bq);
          df_fma_acc(a2, Aq[2 * rstep], bq);
          df_fma_acc(a3, Aq[3 * rstep], bq);
        }
        Gs[r * N + c] = df_finish(a0);
        Gs[(r + rstep) * N + c] = df_finish(a1);
        Gs[(r + 2 * rstep) * N + c] = df_finish(a2);
        Gs[(r + 3 * rstep) * N + c] = df_finish(a3);
      }
      for (; r < N; r += rstep) {
        df2 acc = Gs[r * N + c];
        for (int q = 0; q < m; ++q) df_fma_acc(acc, A_[q * N + r], B_[q * N + c]);
        Gs[r * N + c] = df_finish(acc);
      }
    }
  }
}

__global__ void __launch_bounds__(kThreadsDf, 2) k_flip_df(const FlipArgs<df2> f) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int s_accept[2];  // by attempt parity: see the loop
  __shared__ df2 s_coef[2];
  __shared__ double s_sign;
  __shared__ unsigned long long s_cnt[3];

  const int c = blockIdx.x;
  const int N = f.N, KK = f.kk;
  const long long NN = (long long)N * N;
  const int ns = f.ns;
  df2* Ap = (df2*)smraw;
  df2* Bp = Ap + ns * KK * N;
  df2* dg = Bp + ns * KK * N;         // running diagonal of G^, [ns][N]
  df2* Gs = dg + ns * N;
  // uniforms as FP32 pairs: u = x0 * 2^-32 has at most 32 significant bits, so the pair
  // holds it exactly
  df2* udf = (df2*)(((uintptr_t)(Gs + (f.g_in_smem ? ns * NN : 0)) + 15) & ~(uintptr_t)15);
  int8_t* sl = (int8_t*)(udf + N);

  df2* Gg = f.G + (long long)c * ns * NN;
  df2* G = f.g_in_smem ? Gs : Gg;
  int8_t* fl = f.fields + ((long long)c * f.L + f.l) * N;
  // Philox counter words of this chain: its global index, and sweeps since its start
  const uint32_t gchain = (uint32_t)(f.chain_id ? f.chain_id[c] : f.chain_offset + c);
  const uint32_t sweep = (uint32_t)((f.ctr ? f.ctr[0] : (long long)f.sweep) -
                                    (f.sweep_base ? f.sweep_base[c] : 0));
  const uint8_t* rp = f.replay ? f.replay + ((long long)c * f.L + f.l) * N : nullptr;

  for (int i = threadIdx.x; i < N; i += blockDim.x) {
    sl[i] = fl[i];
    uint32_t ctr[4] = {(uint32_t)(f.l * N + i), sweep, gchain, kTagFlip};
    philox4x32_10(ctr, f.key0, f.key1);
    udf[i] = df_from_double((double)ctr[0] * 2.3283064365386962890625e-10);  // 2^-32
  }
  if (f.g_in_smem)
    for (long long e = threadIdx.x; e < ns * NN; e += blockDim.x) Gs[e] = Gg[e];
  if (threadIdx.x == 0) {
    s_sign = f.sign[c];
    s_cnt[0] = s_cnt[1] = s_cnt[2] = 0;
  }
  __syncthreads();
  for (int i = threadIdx.x; i < ns * N; i += blockDim.x) {
    const int sp = i / N, r = i % N;
    dg[i] = G[sp * NN + (long long)r * N + r];
  }
  __syncthreads();

  // Per attempt: every thread first computes its entries of column i and row i of G^ into
  // panel slot m (they do not depend on the decision) while the last thread evaluates the
  // ratio; after the barrier an acceptance only scales the column by the coefficient and
  // updates the running diagonal, and a rejection leaves slot m to the next attempt. The
  // ratio's latency thus hides behind the panel products instead of adding to them. Flags
  // are double-buffered by attempt parity (see k_flip).
  const df2 one{1.f, 0.f};
  const int rt = kPanelThreads;   // the ratio thread: lane 0 of the last warp
  // entry t of the panels (kind 0: column i of G^, kind 1: row i; spin sp; index r)
  auto panel_entry = [&](int t, int i, int m) {
    const int kind = t / (ns * N), e = t - kind * ns * N;
    const int sp = e / N, r = e % N;
    const df2* Gsp = G + sp * NN;
    const df2* A_ = Ap + sp * KK * N;
    const df2* B_ = Bp + sp * KK * N;
    if (kind == 0) {   // column i of G^, row r
      df2 ca = Gsp[(long long)r * N + i];
      for (int q = 0; q < m; ++q) df_fma_acc(ca, A_[q * N + r], B_[q * N + i]);
      df2 v = df_neg(df_finish(ca));
      if (r == i) v = df_add(v, one);
      if (NMC_DCHECK(m < KK && sp < ns && r < N, 101))
        Ap[(sp * KK + m) * N + r] = v;        // times the coefficient once accepted
    } else {           // row i of G^, column r
      df2 rb = Gsp[(long long)i * N + r];
      for (int q = 0; q < m; ++q) df_fma_acc(rb, A_[q * N + i], B_[q * N + r]);
      if (NMC_DCHECK(m < KK && sp < ns && r < N, 102)) Bp[(sp * KK + m) * N + r] = df_finish(rb);
    }
  };
  // When one pass of the panel threads covers both panels (2 ns N <= 256, so N <= 64), each
  // thread keeps one entry for the whole slice: its column or row, spin and index are
  // computed once here instead of by integer divisions at every attempt.
  const bool one_pass = 2 * ns * N <= kPanelThreads;
  const int tp = threadIdx.x;
  const bool has_entry = tp < 2 * ns * N && tp < kPanelThreads;
  const int p_kind = has_entry ? tp / (ns * N) : 0;
  const int p_e = tp - p_kind * ns * N;
  const int p_sp = has_entry ? p_e / N : 0, p_r = has_entry ? p_e % N : 0;
  const df2* const pG = G + p_sp * NN;
  const df2* const pA = Ap + p_sp * KK * N;
  const df2* const pB = Bp + p_sp * KK * N;
  df2* const pOut = (p_kind == 0 ? Ap : Bp) + p_sp * KK * N + p_r;   // + m N
  int m = 0;
  for (int i = 0; i < N; ++i) {
    if (one_pass) {
      if (has_entry) {
        // the same operations as panel_entry, on this thread's fixed entry
        if (p_kind == 0) {   // column i of G^, row p_r
          df2 ca = pG[(long long)p_r * N + i];
          for (int q = 0; q < m; ++q) df_fma_acc(ca, pA[q * N + p_r], pB[q * N + i]);
          df2 v = df_neg(df_finish(ca));
          if (p_r == i) v = df_add(v, one);
          if (NMC_DCHECK(m < KK, 104)) pOut[m * N] = v;
        } else {             // row i of G^, column p_r
          df2 rb = pG[(long long)i * N + p_r];
          for (int q = 0; q < m; ++q) df_fma_acc(rb, pA[q * N + i], pB[q * N + p_r]);
          if (NMC_DCHECK(m < KK, 105)) pOut[m * N] = df_finish(rb);
        }
      }
    } else if (threadIdx.x < kPanelThreads) {
      for (int t = threadIdx.x; t < 2 * ns * N; t += kPanelThreads) panel_entry(t, i, m);
    }
    if (threadIdx.x == rt) {
      const int s = sl[i];
      const df2 gu = dg[i];
      const df2 du = (s > 0) ? f.dm2 : f.dp2;  // e^{-2 lam s} - 1
      const df2 dd = (s > 0) ? f.dp2 : f.dm2;  // e^{+2 lam s} - 1
      const df2 Ru = df_add(one, df_mul(du, df_add(one, df_neg(gu))));
      // spin down: 1 - G^dn_ii, or G^up_ii when G_dn = I - P G_up^T P
      const df2 omd = ns == 2 ? df_add(one, df_neg(dg[N + i])) : gu;
      const df2 Rd = df_add(one, df_mul(dd, omd));
      const df2 R = df_mul(Ru, Rd);
      const df2 diff = df_add(udf[i], df_neg(df_abs(R)));
      const float margin = 1e-10f * (fabsf(R.hi) + 1.f);
      bool mine;
      double Rsign = R.hi;
      if (fabsf(diff.hi) > margin) {
        mine = diff.hi < 0.f;
      } else {  // certified FP64 evaluation from the same G^_ii
        const double g64u = df_to_double(gu);
        const double omd64 = ns == 2 ? 1.0 - df_to_double(dg[N + i]) : g64u;
        const double d64u = (s > 0) ? f.dm : f.dp, d64d = (s > 0) ? f.dp : f.dm;
        const double R64 = (1.0 + d64u * (1.0 - g64u)) * (1.0 + d64d * omd64);
        mine = df_to_double(udf[i]) < fabs(R64);
        Rsign = R64;
      }
      bool acc_flip = mine;
      if (rp) {
        acc_flip = rp[i] != 0;
        if (acc_flip != mine) s_cnt[2]++;
      }
      s_cnt[0]++;
      s_accept[i & 1] = acc_flip ? 1 : 0;
      if (acc_flip) {
        s_coef[0] = df_neg(df_mul(du, df_rcp(Ru)));
        s_coef[1] = df_neg(df_mul(dd, df_rcp(Rd)));
        if (Rsign < 0.0) s_sign = -s_sign;
        s_cnt[1]++;
        sl[i] = (int8_t)(-s);
      }
    }
    __syncthreads();
    if (s_accept[i & 1]) {
      if (one_pass) {   // thread t < ns N: spin t / N, index t % N (ns N <= 128 <= threads)
        if (tp < ns * N && NMC_DCHECK(m < KK, 103)) {
          const int sp = tp >= N ? 1 : 0, r = tp - sp * N;
          const long long o = (long long)(sp * KK + m) * N + r;
          const df2 a = df_mul(s_coef[sp], Ap[o]);
          Ap[o] = a;
          dg[tp] = df_add(dg[tp], df_mul(a, Bp[o]));
        }
      } else {
        for (int t = threadIdx.x; t < ns * N; t += blockDim.x) {
          const int sp = t / N, r = t % N;
          const long long o = (long long)(sp * KK + m) * N + r;
          if (!NMC_DCHECK(m < KK, 103)) continue;
          const df2 a = df_mul(s_coef[sp], Ap[o]);
          Ap[o] = a;
          dg[t] = df_add(dg[t], df_mul(a, Bp[o]));
        }
      }
      ++m;
      __syncthreads();
      if (m == KK) {
        flush_df(G, Ap, Bp, m, N, KK, NN, ns);
        m = 0;
        __syncthreads();
        for (int j = threadIdx.x; j < ns * N; j += blockDim.x) {
          const int sp = j / N, r = j % N;
          dg[j] = G[sp * NN + (long long)r * N + r];
        }
        __syncthreads();
      }
    }
  }
  if (m > 0) {
    flush_df(G, Ap, Bp, m, N, KK, NN, ns);
    __syncthreads();
  }
  if (f.g_in_smem)
    for (long long e = threadIdx.x; e < ns * NN; e += blockDim.x) Gg[e] = Gs[e];
  for (int i = threadIdx.x; i < N; i += blockDim.x) fl[i] = sl[i];
  if (threadIdx.x == 0) {
    f.sign[c] = s_sign;
    f.counts[3 * c + 0] += s_cnt[0];
    f.counts[3 * c + 1] += s_cnt[1];
    f.counts[3 * c + 2] += s_cnt[2];
  }
}

// ---------------------------------------------------------------------------- blocks of sites
// One slice in blocks of up to 16 sites (Nukala et al., Phys. Rev. B 80, 195111 (2009); Gull et
// al., Phys. Rev. B 83, 075122 (2011)): the decisions of a block need only the 16 x 16 submatrix of
// G^ at its sites. Four warps take them, each holding four of the submatrix's rows for both spins
// (half a warp per spin, lane j column j):
//   R^sigma = 1 + Delta^sigma (1 - G^_ii),   accept iff u < |R^up R^dn|,
//   on acceptance G^ += x y^T with x_r = G^_{ri} - delta_ri, y_j = (Delta / R^sigma) G^_{ij}.
// Until the next acceptance G^ does not change, so all remaining sites are decided at once, one per
// lane, and the first accepted one is next: a rejection costs nothing. A decision is taken in FP32
// when |u - |R|| exceeds a bound on FP32's error, and in FP64 from the same G^_ii otherwise, so it is
// the FP64 decision. Then all threads form the x and y of the block's accepted flips over all N
// sites, one entry of every vector per thread (a triangular recurrence with the submatrix's own x and
// y as coefficients), and the block is folded into G.
//
// The fold G += sum_q x_q y_q^T is one k-step of 16 on the tensor cores by exact FP16 digits
// (fold16.cuh), cut straight from the registers the vectors were formed in.
// Without tensor cores (FP32X2) the vectors go through shared memory to the FP32-pair loop.
//
// One slice, us, one flip at a time (k_flip, k_flip_df) -> here, two thirds of the flips accepted (U = 4):
//   64 sites x 256 chains, both spins: FP32 pairs 133 -> 90, FP64 356 -> 181; a third of them (U = 8): 104 -> 74,
//   244 -> 137; 72 x 1024, one spin, pairs: 420 -> 307; 256 x 32: 2751 -> 444; 100 x 64: 315 -> 140;
//   16 x 256 in FP64: 50 -> 37. (FP32X2: see flip_slice.)
// What bounds it at 64 x 256 (two CTAs per SM): latency. Of a slice's 146k cycles (44% accepted) the decisions take
// 45k (28 acceptances of some 1500: two ratios, a reciprocal and four rows' updates in a dependent
// chain), the folds 47k (of which the MMAs' issue is 23k), the digits 24k, the vectors 13k. In FP64
// the pipe's one instruction per 20 cycles bounds vectors and fold sums.
constexpr int kSites = kFoldK;             // sites per block
enum FoldKind { kFoldTensor, kFoldPairs };

template <typename T> struct Arith;
template <> struct Arith<df2> {
  static __device__ __forceinline__ df2 zero() { return df_zero(); }
  static __device__ __forceinline__ df2 one() { return df2{1.f, 0.f}; }
  static __device__ __forceinline__ float top(df2 a) { return a.hi; }
  static __device__ __forceinline__ double wide(df2 a) { return df_to_double(a); }
  static __device__ __forceinline__ df2 mul(df2 a, df2 b) { return df_mul(a, b); }
  static __device__ __forceinline__ df2 sub(df2 a, df2 b) { return df_add(a, df_neg(b)); }
  static __device__ __forceinline__ df2 add(df2 a, df2 b) { return df_add(a, b); }
  static __device__ __forceinline__ void fma_acc(df2& c, df2 a, df2 b) { df_fma_acc(c, a, b); }
  static __device__ __forceinline__ df2 finish(df2 a) { return df_finish(a); }
  static __device__ __forceinline__ df2 div(df2 a, df2 b) { return df_div(a, b); }
};
template <> struct Arith<double> {
  static __device__ __forceinline__ double zero() { return 0.0; }
  static __device__ __forceinline__ double one() { return 1.0; }
  static __device__ __forceinline__ float top(double a) { return (float)a; }
  static __device__ __forceinline__ double wide(double a) { return a; }
  static __device__ __forceinline__ double mul(double a, double b) { return a * b; }
  static __device__ __forceinline__ double sub(double a, double b) { return a - b; }
  static __device__ __forceinline__ double add(double a, double b) { return a + b; }
  static __device__ __forceinline__ void fma_acc(double& c, double a, double b) { c = fma(a, b, c); }
  static __device__ __forceinline__ double finish(double a) { return a; }
  // (two sweeps of 64 sites x 256 chains: 31.2 ms with the division, 30.5 so)
  static __device__ __forceinline__ double div(double a, double b) { return quotient(a, b); }
};

// a load that does not look into the SM's own cache
__device__ __forceinline__ double ld_l2(const double* p) { return __ldcg(p); }
__device__ __forceinline__ df2 ld_l2(const df2* p) {
  const float2 v = __ldcg((const float2*)p);
  return df2{v.x, v.y};
}

template <typename T> __device__ __forceinline__ T delta(const FlipArgs<T>& f, bool plus);
template <> __device__ __forceinline__ df2 delta<df2>(const FlipArgs<df2>& f, bool plus) { return plus ? f.dp2 : f.dm2; }
template <> __device__ __forceinline__ double delta<double>(const FlipArgs<double>& f, bool plus) { return plus ? f.dp : f.dm; }
// G[s][r][c] += sum_q x[s][q][r] y[s][q][c] on the FP32 pipe: four rows at a time, four independent
// chains per y read
template <typename T>
__device__ void fold_pairs(T* G, const T* pan, int m, int N, int ns, long long sG, int ld) {
  const int nthr = blockDim.x, c0 = threadIdx.x % N, r0 = threadIdx.x / N;
  const int rstep = nthr >= N ? nthr / N : 1;
  if (nthr >= N && r0 >= rstep) return;
  for (int s = 0; s < ns; ++s) {
    const T* x = pan + (long long)s * kSites * N;
    const T* y = pan + (long long)(ns + s) * kSites * N;
    T* Gp = G + s * sG;
    for (int c = c0; c < N; c += nthr >= N ? N : nthr)
      for (int r = nthr >= N ? r0 : 0; r < N; r += 4 * rstep) {
        T a[4];
#pragma unroll
        for (int i = 0; i < 4; ++i)
          a[i] = r + i * rstep < N ? Gp[(long long)(r + i * rstep) * ld + c] : Arith<T>::zero();
        for (int q = 0; q < m; ++q) {
          const T b = y[q * N + c];
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (r + i * rstep < N) Arith<T>::fma_acc(a[i], x[q * N + r + i * rstep], b);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (r + i * rstep < N) Gp[(long long)(r + i * rstep) * ld + c] = Arith<T>::finish(a[i]);
      }
  }
}

// the deciding warps, 4 rows of the block each
constexpr int kDecide = kSites / 4;
__device__ __forceinline__ void bar_decide() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kDecide) : "memory"); }

// stage arrays of one block, in shared memory
template <typename T>
struct BlockStage {
  T S[2][kSites][kSites];     // [spin]: G^ at the block's sites, while they are decided
  T x[2][kSites][kSites];     // [spin][accepted flip q][block row]: x_q at the block's later sites
  T y[2][kSites][kSites];     // [spin][q][block column]
  T c[2][kSites];             // Delta / R^sigma of q
  int site[kSites];           // block index of q
  int m[2];                   // accepted flips, by block parity: see the loop
};

// The decisions of the block of kb sites from i0 on, by the first kDecide warps: entry(s, t, j) is G^'s
// row t and column j of the block for spin s. Leaves the accepted flips in st, their number in
// st.m[slot], and the flipped signs in sl.
template <typename T, typename F>
__device__ __forceinline__ void decide_block(const FlipArgs<T>& f, BlockStage<T>& st, int i0, int kb, int slot,
                                             const unsigned* u, int8_t* sl, const uint8_t* rp, double& sign,
                                             unsigned long long& n_acc, unsigned long long& n_dis, F entry) {
  typedef Arith<T> A;
  const int ns = f.ns, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sp = ns == 2 ? lane >> 4 : 0, j = lane & 15;   // this lane's spin and column
  const float fm = (float)f.dm, fp = (float)f.dp;
  T* S = &st.S[sp][0][j];   // this lane's column: row t at S[t * kSites]
#pragma unroll
  for (int t = 4 * warp; t < 4 * warp + 4; ++t)
    S[t * kSites] = t < kb && j < kb ? entry(sp, t, j) : A::zero();
  const int jj = min(j, kb - 1), s_j = sl[i0 + jj];   // (read before the first flip's write, see the barrier)
  const bool pos = s_j > 0;
  const unsigned u_j = u[i0 + jj];
  const float uf = (float)u_j * 0x1p-32f, du = pos ? fm : fp, dd = pos ? fp : fm;
  bar_decide();
  int m = 0;
  for (int lo = 0; lo < kb;) {   // sites below lo are decided
    // every remaining site as if it were the next: lane j site j. (A faster warp may already update its rows
    // below the flip that all warps are about to find: only entries of sites beyond that flip change, and
    // neither the first accepted site nor anything taken from it depends on them.)
    const T gu = st.S[0][jj][jj], gd = ns == 2 ? st.S[1][jj][jj] : gu;
    const float hu = 1.f - A::top(gu), hd = ns == 2 ? 1.f - A::top(gd) : A::top(gu);
    const float R32 = (1.f + du * hu) * (1.f + dd * hd);
    // FP32's error: a few 2^-24 of (1 + |du| (1 + |g|)) (1 + |dd| (1 + |g|))
    const float bound = 2e-6f * (1.f + fabsf(du) * (1.f + fabsf(hu))) *
                        (1.f + fabsf(dd) * (1.f + fabsf(hd)));
    const bool open = j >= lo && j < kb;
    bool mine = uf < fabsf(R32), neg = R32 < 0.f;
    if (open && (rp || !(fabsf(uf - fabsf(R32)) > bound))) {   // in FP64, from the same G^_ii
      const double g64 = A::wide(gu), h64 = ns == 2 ? 1.0 - A::wide(gd) : g64;
      const double R = (1.0 + (pos ? f.dm : f.dp) * (1.0 - g64)) *
                       (1.0 + (pos ? f.dp : f.dm) * h64);
      mine = (double)u_j * 0x1p-32 < fabs(R);
      neg = R < 0.0;
    }
    bool take = mine;
    if (rp) take = rp[i0 + jj] != 0;
    const unsigned takes = __ballot_sync(0xffffffffu, open && take) & 0xffffu;
    const int b = takes ? __ffs(takes) - 1 : kb;      // the next accepted site; the rest up to it are rejected
    if (rp)
      n_dis += __popc(__ballot_sync(0xffffffffu, open && j <= b && take != mine) & 0xffffu);
    if (b == kb) break;
    ++n_acc;
    if (__shfl_sync(0xffffffffu, (int)neg, b)) sign = -sign;
    const bool posb = __shfl_sync(0xffffffffu, (int)pos, b);
    // y = (Delta / R) row of G^, on every lane its entry
    const T d = posb == (sp == 0) ? delta<T>(f, false) : delta<T>(f, true);
    const T R = A::add(A::one(), A::mul(d, A::sub(A::one(), st.S[sp][b][b])));
    const T q = A::div(d, R);
    const T y = A::mul(q, S[b * kSites]);
    if (!NMC_DCHECK(m < kSites && b < kSites, 121)) break;
    if (warp == 0) {
      st.y[sp][m][j] = y;
      st.c[sp][m] = q;
      if (lane == 0) {
        st.site[m] = b;
        sl[i0 + b] = (int8_t)(posb ? -1 : 1);
      }
    }
    // this warp's rows below b: G^ += x y^T, x the column of site b
    if (4 * warp + 3 > b) {
      T z[4], x[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        x[k] = st.S[sp][4 * warp + k][b];
        z[k] = S[(4 * warp + k) * kSites];
      }
      __syncwarp();
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        A::fma_acc(z[k], x[k], y);
        if (4 * warp + k > b) {
          S[(4 * warp + k) * kSites] = A::finish(z[k]);
          st.x[sp][m][4 * warp + k] = x[k];
        }
      }
    }
    ++m;
    lo = b + 1;
    bar_decide();
  }
  if (threadIdx.x == 0) st.m[slot] = m;
}

// x_q[r] (kind 0) or y_q[r] (kind 1) of the block's m flips for spin sv; rel: r less the block's first
// site; entry(s): G's entry at row r and the block's column s (kind 1: row s and column r)
template <typename T, typename F>
__device__ __forceinline__ void block_vectors(const BlockStage<T>& st, int kind, int sv, int rel, int m,
                                              T (&v)[kSites], F entry) {
  typedef Arith<T> A;
  const T* coef = kind ? &st.x[sv][0][0] : &st.y[sv][0][0];
  T g[kSites];
#pragma unroll
  for (int p = 0; p < kSites; ++p) g[p] = p < m ? entry(st.site[p]) : A::zero();
#pragma unroll
  for (int p = 0; p < kSites; ++p) {
    v[p] = A::zero();
    if (p >= m) continue;
    const int s = st.site[p];
    T z = g[p];
#pragma unroll
    for (int q = 0; q < p; ++q) A::fma_acc(z, coef[q * kSites + s], v[q]);
    z = A::finish(z);
    if (kind) z = A::mul(st.c[sv][p], z);
    else if (rel == s) z = A::sub(z, A::one());
    v[p] = z;
  }
}

template <typename T>
__host__ __device__ inline size_t block_smem(int N, int ns, bool g_in_smem, int fold, int ld) {
  const int Np = (N + 15) & ~15;
  size_t b = g_in_smem ? (size_t)ns * N * ld * sizeof(T) : 0;
  b += fold == kFoldTensor ? (size_t)2 * kFDig * Np * 32 + 2 * Np * sizeof(int)
                           : (size_t)2 * ns * kSites * N * sizeof(T);
  b += sizeof(BlockStage<T>) + (size_t)N * 4 + ((N + 15) & ~15);
  return b + 64;
}

// GS: G held in shared memory
template <typename T, int FOLD, int THREADS, bool GS>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? 2 : 1)
k_flip_block(const FlipArgs<T> f, int kb_max) {
  typedef Arith<T> A;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int c = blockIdx.x, N = f.N, ns = f.ns, Np = (N + 15) & ~15;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int ld = GS ? N + 2 : N;   // (rows of a column read on different banks)
  const long long NN = (long long)N * N, sG = GS ? (long long)N * ld : NN;
  T* Gs = (T*)smraw;
  T* Gg = f.G + (long long)c * ns * NN;
  T* G;
  if constexpr (GS) G = Gs;
  else G = Gg;
  unsigned char* dig = smraw + (GS ? (size_t)ns * N * ld * sizeof(T) : 0);
  T* pan = (T*)dig;                                  // kFoldPairs: [x, y][ns][16][N]
  int* ev = (int*)(dig + (size_t)2 * kFDig * Np * 32);   // kFoldTensor: exponents of x rows, y columns
  // (every part a multiple of 16 bytes: N is even)
  BlockStage<T>& st = *(BlockStage<T>*)(dig + (FOLD == kFoldTensor ? (size_t)2 * kFDig * Np * 32 + 2 * Np * sizeof(int)
                                                                   : (size_t)2 * ns * kSites * N * sizeof(T)));
  unsigned* u = (unsigned*)(&st + 1);                // Philox words: u_i = word 2^-32
  int8_t* sl = (int8_t*)(u + N);

  int8_t* fl = f.fields + ((long long)c * f.L + f.l) * N;
  const uint32_t gchain = (uint32_t)(f.chain_id ? f.chain_id[c] : f.chain_offset + c);
  const uint32_t sweep = (uint32_t)((f.ctr ? f.ctr[0] : (long long)f.sweep) -
                                    (f.sweep_base ? f.sweep_base[c] : 0));
  const uint8_t* rp = f.replay ? f.replay + ((long long)c * f.L + f.l) * N : nullptr;
  for (int i = tid; i < N; i += THREADS) {
    sl[i] = fl[i];
    uint32_t ctr[4] = {(uint32_t)(f.l * N + i), sweep, gchain, kTagFlip};
    philox4x32_10(ctr, f.key0, f.key1);
    u[i] = ctr[0];
  }
  if (GS)
    for (int e = tid; e < ns * N * (N / 2); e += THREADS) {   // two entries at a time (N is even)
      const int r = e / (N / 2);
      *(float4*)(Gs + 2 * e + r * (ld - N)) = *(const float4*)(Gg + 2 * e);
    }
  double sign = 1.0;
  unsigned long long n_acc = 0, n_dis = 0;
  __syncthreads();

  // (A block without a flip has one barrier: thread 0 may then write the next block's count while
  // slower warps still read this one's, hence two slots. It writes this slot again only after every
  // warp has passed the next block's barrier.)
  for (int i0 = 0, blk = 0; i0 < N; i0 += kb_max, ++blk) {
    const int kb = min(kb_max, N - i0);
    if (warp < kDecide)
      decide_block(f, st, i0, kb, blk & 1, u, sl, rp, sign, n_acc, n_dis,
                   [&](int s, int t, int k) { return G[s * sG + (long long)(i0 + t) * ld + i0 + k]; });
    __syncthreads();
    const int m = st.m[blk & 1];
    if (m > 0) {
      // ---------------------------------------------------------- the vectors over all sites
      auto vectors = [&](int kind, int sv, int r, T (&v)[kSites]) {
        const T* base = G + sv * sG + (kind ? (long long)i0 * ld + r : (long long)r * ld + i0);
        const int step = kind ? ld : 1;
        block_vectors(st, kind, sv, r - i0, m, v, [&](int s) { return base[(long long)s * step]; });
      };
      if constexpr (FOLD == kFoldPairs) {
        for (int t = tid; t < 2 * ns * N; t += THREADS) {
          const int kind = t / (ns * N), e = t - kind * ns * N, sv = e / N, r = e - sv * N;
          T v[kSites];
          vectors(kind, sv, r, v);
#pragma unroll
          for (int p = 0; p < kSites; ++p)
            if (p < m) pan[((kind * ns + sv) * kSites + p) * N + r] = v[p];
        }
        __syncthreads();
        fold_pairs(G, pan, m, N, ns, sG, ld);
      } else {
        // digits of one spin at a time: both would not leave room for a second CTA on the SM
        const int stride = Np * 32;
        const bool once = 2 * ns * N <= THREADS;   // every thread one entry of one spin
        T v[kSites];
        int E = Digits<T>::kExpMin;
        auto limit = [&] {
          E = Digits<T>::kExpMin;
#pragma unroll
          for (int p = 0; p < kSites; ++p) E = max(E, Digits<T>::expo(v[p]));
        };
        const int k0 = tid / (ns * N), e0 = tid - k0 * ns * N, s0 = e0 / N, r0 = e0 - s0 * N;
        if (once && k0 < 2) {
          vectors(k0, s0, r0, v);
          limit();
        }
        for (int sf = 0; sf < ns; ++sf) {
          if (sf) __syncthreads();   // the other spin's digits are read
          if (once) {
            if (k0 < 2 && s0 == sf) {
              ev[k0 * Np + r0] = Digits<T>::scale(E);
              cut16<T>(v, E, dig + k0 * kFDig * stride, r0, stride);
            }
          } else {
            for (int t = tid; t < 2 * N; t += THREADS) {
              const int kind = t / N, r = t - kind * N;
              vectors(kind, sf, r, v);
              limit();
              ev[kind * Np + r] = Digits<T>::scale(E);
              cut16<T>(v, E, dig + kind * kFDig * stride, r, stride);
            }
          }
          __syncthreads();
          T* Gf = G + sf * sG;
          const unsigned dbase = (unsigned)__cvta_generic_to_shared(dig);
          fold_tiles<T>([&](int r) { return Gf + (long long)r * ld; }, dbase, stride, ev,
                        dbase + kFDig * stride, stride, ev + Np, N, N, true, warp, THREADS / 32);   // (N is even)
        }
      }
      __syncthreads();
    }
  }
  if (GS)
    for (int e = tid; e < ns * N * (N / 2); e += THREADS) {
      const int r = e / (N / 2);
      *(float4*)(Gg + 2 * e) = *(const float4*)(Gs + 2 * e + r * (ld - N));
    }
  for (int i = tid; i < N; i += THREADS) fl[i] = sl[i];
  if (tid == 0) {
    f.sign[c] *= sign;
    f.counts[3 * c + 0] += (unsigned long long)N;
    f.counts[3 * c + 1] += n_acc;
    f.counts[3 * c + 2] += n_dis;
  }
}

// The same for G in global memory and fewer chains than SMs: a cluster of CTAs per chain. Every CTA takes
// all decisions (from the same G, so the same ones), forms and folds the rows of its share of 16-row
// tiles, and forms the columns of the same share, whose digits it writes to every CTA of the cluster.
// Each entry sees the operations of k_flip_block in the same order. The barriers do not depend on what
// was decided. 256 sites x 32 chains, us (44% accepted): one CTA per chain 966, two 557, four 391; eight (x 16 chains)
// 585 for four's 383. 100 x 64 with two 118 against 133 with G in shared memory; 64 x 32 59 against 55,
// hence kClusterMinN where shared memory would do.
constexpr int kClusterMinN = 96;

template <typename T>
__host__ __device__ inline size_t cluster_smem(int N, int ns, int cs) {
  const int tiles = (N + 15) >> 4, own = (tiles + cs - 1) / cs * 16, Np = tiles * 16;
  return (size_t)ns * (own + Np) * (kFDig * 32 + 4) + sizeof(BlockStage<T>) + (size_t)N * 4 + ((N + 15) & ~15) + 64;
}

template <typename T>
__global__ void __launch_bounds__(512, 1)
k_flip_cluster(const FlipArgs<T> f, int kb_max) {
  constexpr int THREADS = 512;
  extern __shared__ __align__(16) unsigned char smraw[];
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int c = blockIdx.x / cs, N = f.N, ns = f.ns, tiles = (N + 15) >> 4, Np = tiles * 16;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int own = (tiles + cs - 1) / cs * 16;                    // rows of the largest share
  const int r0 = tiles * rank / cs * 16, nr = max(min(tiles * (rank + 1) / cs * 16, N) - r0, 0);
  const long long NN = (long long)N * N;
  T* G = f.G + (long long)c * ns * NN;
  const int xs = own * 32, ys = Np * 32;                         // bytes per digit
  unsigned char* xd = smraw;                                     // [spin][digit][own rows]
  unsigned char* yd = xd + (size_t)ns * kFDig * xs;              // [spin][digit][columns]
  int* xe = (int*)(yd + (size_t)ns * kFDig * ys);
  int* ye = xe + ns * own;
  BlockStage<T>& st = *(BlockStage<T>*)(ye + ns * Np);
  unsigned* u = (unsigned*)(&st + 1);
  int8_t* sl = (int8_t*)(u + N);

  int8_t* fl = f.fields + ((long long)c * f.L + f.l) * N;
  const uint32_t gchain = (uint32_t)(f.chain_id ? f.chain_id[c] : f.chain_offset + c);
  const uint32_t sweep = (uint32_t)((f.ctr ? f.ctr[0] : (long long)f.sweep) -
                                    (f.sweep_base ? f.sweep_base[c] : 0));
  const uint8_t* rp = f.replay ? f.replay + ((long long)c * f.L + f.l) * N : nullptr;
  for (int i = tid; i < N; i += THREADS) {
    sl[i] = fl[i];
    uint32_t ctr[4] = {(uint32_t)(f.l * N + i), sweep, gchain, kTagFlip};
    philox4x32_10(ctr, f.key0, f.key1);
    u[i] = ctr[0];
  }
  double sign = 1.0;
  unsigned long long n_acc = 0, n_dis = 0;
  cl.sync();   // (no CTA writes the fields or another's memory before all have begun)

  for (int i0 = 0, blk = 0; i0 < N; i0 += kb_max, ++blk) {
    const int kb = min(kb_max, N - i0);
    if (warp < kDecide)   // (rows of other shares: past the L1)
      decide_block(f, st, i0, kb, blk & 1, u, sl, rp, sign, n_acc, n_dis,
                   [&](int s, int t, int k) { return ld_l2(G + s * NN + (long long)(i0 + t) * N + i0 + k); });
    __syncthreads();
    const int m = st.m[blk & 1];
    if (m > 0) {
      for (int t = tid; t < 2 * ns * nr; t += THREADS) {
        const int kind = t / (ns * nr), e = t - kind * ns * nr, sv = e / nr, k = e - sv * nr, r = r0 + k;
        const T* base = G + sv * NN + (kind ? (long long)i0 * N + r : (long long)r * N + i0);
        const int step = kind ? N : 1;
        T v[kSites];
        block_vectors(st, kind, sv, r - i0, m, v, [&](int s) { return ld_l2(base + (long long)s * step); });
        int E = Digits<T>::kExpMin;
#pragma unroll
        for (int p = 0; p < kSites; ++p) E = max(E, Digits<T>::expo(v[p]));
        if (kind == 0) {
          xe[sv * own + k] = Digits<T>::scale(E);
          cut16<T>(v, E, xd + (size_t)sv * kFDig * xs, k, xs);
        } else {
          for (int q = 0; q < cs; ++q) cl.map_shared_rank(ye, q)[sv * Np + r] = Digits<T>::scale(E);
          unsigned char* dst = yd + (size_t)sv * kFDig * ys;
          cut16_to(v, E, [&](int s, int h, uint4 w) {
            for (int q = 0; q < cs; ++q)
              *reinterpret_cast<uint4*>(cl.map_shared_rank(dst, q) + s * ys + digit_off(r, h)) = w;
          });
        }
      }
    }
    cl.sync();
    if (m > 0 && nr > 0)
      for (int sv = 0; sv < ns; ++sv) {
        T* Gf = G + sv * NN + (long long)r0 * N;
        fold_tiles<T>([&](int r) { return Gf + (long long)r * N; },
                      (unsigned)__cvta_generic_to_shared(xd + (size_t)sv * kFDig * xs), xs, xe + sv * own,
                      (unsigned)__cvta_generic_to_shared(yd + (size_t)sv * kFDig * ys), ys, ye + sv * Np,
                      nr, N, true, warp, THREADS / 32);
      }
    __threadfence();
    cl.sync();
  }
  if (rank == 0) {
    for (int i = tid; i < N; i += THREADS) fl[i] = sl[i];
    if (tid == 0) {
      f.sign[c] *= sign;
      f.counts[3 * c + 0] += (unsigned long long)N;
      f.counts[3 * c + 1] += n_acc;
      f.counts[3 * c + 2] += n_dis;
    }
  }
}

}  // namespace

size_t flip_smem_bytes(int N, int kk, size_t elem, int g_in_smem, int ns) {
  size_t b = (size_t)(2 * ns * kk * N + ns * N) * elem;
  if (g_in_smem) b += (size_t)ns * N * N * elem;
  b = (b + 15) & ~(size_t)15;
  b += (size_t)N * sizeof(double) + (size_t)N + 16;
  b += 2 * (size_t)ns * N * sizeof(int) + 16;   // (what nmc_get_dims' delay_k is clamped by)
  return b;
}

namespace {

constexpr size_t kBlockSmem = 226 * 1024;   // (227 KB are available)

template <typename T>
void flip_cluster(const FlipArgs<T>& f, int n_chains, int kb, int cs, cudaStream_t st) {
  allow_max_dynamic_smem((const void*)k_flip_cluster<T>);
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = cs;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(n_chains * cs);
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = cluster_smem<T>(f.N, f.ns, cs);
  cfg.stream = st;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_flip_cluster<T>, f, kb);   // (an error is seen by the launch's next check)
}

// One slice by k_flip_block; false: the vectors of a block do not fit shared memory. G is held
// there when it fits with them. 256 threads, two CTAs per SM, when there are more chains than
// SMs; 512 otherwise. (Neither choice changes a bit of the results.)
template <typename T, int FOLD>
bool flip_block(const FlipArgs<T>& f, int n_chains, cudaStream_t st) {
  size_t bytes = block_smem<T>(f.N, f.ns, true, FOLD, f.N + 2);
  const bool gs = bytes <= kBlockSmem;
  if (!gs) bytes = block_smem<T>(f.N, f.ns, false, FOLD, f.N);
  const int kb = f.kk < kSites ? f.kk : kSites;
  if constexpr (FOLD == kFoldTensor)
    if (!gs || f.N >= kClusterMinN) {
      int cs = 4;
      while (cs > 1 && (n_chains * cs > sm_count() || cluster_smem<T>(f.N, f.ns, cs) > kBlockSmem)) cs >>= 1;
      if (cs > 1) {
        flip_cluster(f, n_chains, kb, cs, st);
        return true;
      }
    }
  if (bytes > kBlockSmem) return false;
  auto run = [&](auto kernel, int threads) {
    allow_max_dynamic_smem((const void*)kernel);
    kernel<<<n_chains, threads, bytes, st>>>(f, kb);
  };
  if (!gs) run(k_flip_block<T, FOLD, 512, false>, 512);
  else if (f.N > 48 && (n_chains <= sm_count() || bytes > kBlockSmem / 2)) run(k_flip_block<T, FOLD, 512, true>, 512);
  else run(k_flip_block<T, FOLD, 256, true>, 256);
  return true;
}

template <typename T>
void flip_old(const FlipArgs<T>& f, int n_chains, cudaStream_t st) {
  const size_t bytes = flip_smem_bytes(f.N, f.kk, sizeof(T), f.g_in_smem, f.ns);
  allow_max_dynamic_smem((const void*)k_flip<T>);
  k_flip<T><<<n_chains, kThreads, bytes, st>>>(f);
}

}  // namespace

template <>
void flip_slice<float>(const FlipArgs<float>& f, int n_chains, cudaStream_t st) {
  flip_old(f, n_chains, st);
}

// Small delays: a block of min(delay, 16) sites holds at most so many accepted flips, but a block's fixed
// costs (its submatrix, the vectors over all sites, the digits) want some five of them; below, one flip at
// a time is faster, while its matrices fit shared memory (FP64: twice to an SM). The line follows the
// delay and delay x sites, not the number of chains, so a chain's results do not depend on those beside it.
// us a slice, one at a time / blocks, 66% accepted, by delay:
//   FP32 pairs   16 sites x 512, delay 1 55 / 141, 4 40 / 61, 8 37 / 44, 12 38 / 45, 16 37 / 36;
//                64 x 256, 1 208 / 544, 4 139 / 204, 6 133 / 155, 8 131 / 126;
//                80 x 200, 3 285 / 537, 5 355 / 361, 8 331 / 259;  100 x 64, 4 317 / 344, 5 326 / 286;
//   FP64         16 x 512, 1 76 / 231, 6 72 / 84, 8 73 / 70;  36 x 256, 1 143 / 440, 6 121 / 125, 8 123 / 114;
//                64 x 256, 1 408 / 1007, 4 324 / 371, 5 326 / 317;  100 x 64, 2 956 / 975, 3 823 / 711;
// With every delay in blocks a whole sweep was up to twice as long as with one flip at a time (16 sites x 1 in
// FP64, delay 1: 2.3 / 4.5 ms a pair).
constexpr int kSingleDelay = 8, kSingleWork = 430;           // FP32 pairs
constexpr int kSingleDelay64 = 6, kSingleWork64 = 300;       // FP64

template <>
void flip_slice<double>(const FlipArgs<double>& f, int n_chains, cudaStream_t st) {
  const bool single = f.kk <= kSingleDelay64 && f.kk * f.N <= kSingleWork64 && f.g_in_smem &&
                      flip_smem_bytes(f.N, f.kk, sizeof(double), 1, f.ns) <= kBlockSmem / 2;
  if (single || !flip_block<double, kFoldTensor>(f, n_chains, st)) flip_old(f, n_chains, st);
}

// FP32X2, without tensor cores: a block's fold costs as much as the folds of single flips, and the vectors come
// on top, so blocks pay only for a few sites, and with both spins above 64 sites, where k_flip_df's 256 threads
// take the panels' entries in several passes, as long as G fits a block's shared memory. us a slice at delay 16,
// one at a time / blocks, 66% accepted, both spins: 16 sites x 256 22.7 / 21.9, 36 x 256 53.9 / 59.0, 64 x 256
// 133 / 154, 72 x 16 159 / 133, 72 x 512 592 / 466 (delay 8: 154 / 140 and 406 / 495), 80 x 200 341 / 311,
// 100 x 64 318 / 275, 112 x 64 398 / 434, 144 x 64 742 / 811, 256 x 32 2742 / 3368; one spin: 72 x 1024
// 422 / 471, 120 x 256 436 / 518.
bool pairs_one_at_a_time(const FlipArgs<df2>& f) {
  if (f.kk <= kSingleDelay && f.kk * f.N <= kSingleWork && f.g_in_smem) return true;
  if (f.tc_fold) return false;
  const bool held = block_smem<df2>(f.N, f.ns, true, kFoldPairs, f.N + 2) <= kBlockSmem;
  return f.N > 24 && !(f.ns == 2 && f.N > 64 && held);
}

template <>
void flip_slice<df2>(const FlipArgs<df2>& f, int n_chains, cudaStream_t st) {
  if (!pairs_one_at_a_time(f) && (f.tc_fold ? flip_block<df2, kFoldTensor>(f, n_chains, st)
                                            : flip_block<df2, kFoldPairs>(f, n_chains, st)))
    return;
  const size_t bytes = flip_smem_bytes(f.N, f.kk, sizeof(df2), f.g_in_smem, f.ns);
  allow_max_dynamic_smem((const void*)k_flip_df);
  k_flip_df<<<n_chains, kThreadsDf, bytes, st>>>(f);
}

NMC_DEBUG_READER(debug_fail_flip)

}  // namespace nmc
