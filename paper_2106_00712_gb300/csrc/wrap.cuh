// Whole-matrix products with constant matrices (wrap.cu).
#pragma once
#include <type_traits>

#include "df.cuh"

namespace nmc {

constexpr int kFragMaxN = 112;   // 7 digits of 112 x 112 entries fill shared memory

// A constant's operand fragments: bytes, and their preparation from M (device, FP64, N x N): vectors
// are M's rows (cols = false: M X) or columns (cols = true: X M); scales: 16 ceil(N / 16) ints.
template <typename T> size_t frag_bytes(int N);
template <typename T>
void prepare_frags(const double* M, int N, bool cols, void* frags, int* scales, cudaStream_t st);

// C = L (S X S^{-1}) R (before) or S^{-1} (L X R) S (after), S = diag(e^{sigma lam s}); no S without
// fields. Matrices contiguous N x N, N even; C may be X. Cd instead of C: FP64 results (no fields after).
template <typename T> struct WrapArgs {
  int N = 0, batch = 0, ns = 2;
  const T* X = nullptr; long long sX = 0;
  T* C = nullptr; double* Cd = nullptr;
  const uint4 *L = nullptr, *R = nullptr; const int *Le = nullptr, *Re = nullptr;   // fragments, scales
  const int8_t* fields = nullptr; long long fstride = 0; bool before = false;
  T e2, em2;              // e^{2 lam}, e^{-2 lam}
};
template <typename T> void wrap_product(const WrapArgs<T>& g, cudaStream_t st);

// X = (L S_w) ... (L S_1) U D (before) or (S_w L) ... (S_1 L) U D (after), S_k of slice l0 + (k - 1) dl
template <typename T> struct ChainArgs {
  int N = 0, batch = 0, ns = 2, w = 0, l0 = 0, dl = 1;
  const double* U = nullptr; long long sU = 0;
  const double* Dv = nullptr; long long sD = 0;
  double* X = nullptr;
  const uint4* L = nullptr; const int* Le = nullptr;
  const int8_t* fields = nullptr; long long fstride = 0; bool before = false;
  T e1, em1;              // e^{lam}, e^{-lam}
  double d1, dm1;         // the same in FP64
};
template <typename T> void chain_product(const ChainArgs<T>& g, cudaStream_t st);

}  // namespace nmc
