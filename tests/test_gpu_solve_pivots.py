"""The stabilized solve's pivots over FP64's whole range, called directly: X diagonal and U the identity, so
that Y = diag(1 / x) exactly, whatever the order of the pivots. Random entries, the largest ones (whose
reciprocals are subnormal) and subnormal ones (whose reciprocals are still finite), for Gauss-Jordan (40
sites), the LU in shared memory with one and two CTAs to an SM, and the LU in global memory."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

PROGRAM = r'''
#include <cmath>
#include <cstdio>
#include <vector>
#include "nmc_internal.cuh"
int main() {
  int bad = 0;
  for (int N : {40, 41, 64, 72, 90, 120, 260}) {
    const size_t NN = (size_t)N * N;
    std::vector<double> X(2 * NN, 0.0), U(2 * NN, 0.0), D(2 * N, 1.0), Y(2 * NN);
    unsigned long long s = 12345 + N;
    auto next = [&] { return (s = s * 6364136223846793005ull + 1442695040888963407ull) >> 11; };
    for (int b = 0; b < 2; ++b)
      for (int i = 0; i < N; ++i) {
        const double m = 1.0 + (double)next() * 0x1p-53;   // [1, 2)
        const int e = (int)(next() % 2040) - 1020;
        double x = ldexp(m, e);
        if (i % 7 == 3) x = ldexp(m, 1022 + (int)(next() & 1));    // the largest
        if (i % 7 == 5) x = ldexp(m, -1023);                       // subnormal
        X[b * NN + (size_t)i * N + i] = next() & 1 ? x : -x;
        U[b * NN + (size_t)i * N + i] = 1.0;
      }
    double *dX, *dU, *dD, *dY, *ws;
    cudaMalloc(&dX, X.size() * 8); cudaMalloc(&dU, U.size() * 8); cudaMalloc(&dD, D.size() * 8);
    cudaMalloc(&dY, Y.size() * 8); cudaMalloc(&ws, 4 * NN * 8);
    cudaMemcpy(dX, X.data(), X.size() * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dU, U.data(), U.size() * 8, cudaMemcpyHostToDevice);
    cudaMemcpy(dD, D.data(), D.size() * 8, cudaMemcpyHostToDevice);
    nmc::solve_stab(dX, dU, (long long)NN, dD, N, dY, ws, N, 2, 0);
    if (cudaMemcpy(Y.data(), dY, Y.size() * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
    for (int b = 0; b < 2; ++b)
      for (int i = 0; i < N; ++i)
        for (int j = 0; j < N; ++j) {
          const double y = Y[b * NN + (size_t)i * N + j], x = X[b * NN + (size_t)i * N + i];
          const double want = i == j ? 1.0 / x : 0.0;
          if (!(y == want) && ++bad <= 8) printf("N %d, entry %d %d: %.17g, not %.17g\n", N, i, j, y, want);
        }
    cudaFree(dX); cudaFree(dU); cudaFree(dD); cudaFree(dY); cudaFree(ws);
  }
  printf("%d differ\n", bad);
  return bad ? 1 : 0;
}
'''


def test_reciprocals_of_pivots(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    from paper_2106_00712_gb300 import build_lib
    nvcc = build_lib._nvcc()
    assert shutil.which(nvcc), nvcc
    src, exe = tmp_path / "pivots.cu", tmp_path / "pivots"
    src.write_text(PROGRAM)
    subprocess.run([nvcc, str(src), "-o", str(exe), "-I", build_lib.CSRC, build_lib.LIB]
                   + build_lib.ARCH + build_lib.NVCC_FLAGS, check=True, timeout=300)
    env = dict(os.environ, LD_LIBRARY_PATH=os.path.dirname(build_lib.LIB))
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, env=env)
    assert r.returncode == 0, r.stdout + r.stderr
