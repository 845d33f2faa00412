"""The flips' quotients, each compiled into a program of its own.

FP64 (csrc/quotient.cuh) against the division: 2^24 pairs of random mantissas over the exponents that it
handles itself, 2^24 over all exponents, and every pair of special values. The quotient before its last
rounding is off by less than 2^-48 units of the last place (derived in the header), so a result other than
the division's has a chance of 2^-47 a pair, and none is expected.

FP32 pairs (df_div of csrc/df.cuh) against the FP64 quotient of the same values: 2^24 random pairs, off by at
most the 2.75 x 2^-46 derived there (and the reference's 2^-53) and, where the quotient's low part is
subnormal, three products' and a sum's roundings of 2^-150; and divisors between 2^126 and the largest,
where the FP32 reciprocal has some 22 bits: 2^-20."""
import os
import shutil
import subprocess

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cstdio>
#include <cstring>
#include "nmc_internal.cuh"
#include "quotient.cuh"
using namespace nmc;
__device__ const double special[] = {0.0, -0.0, 1.0, -3.0, 4.9e-324, 2.2e-308, -2.3e-308, 1e-300, 5.07e-116,
                                     5.08e-116, 3.93e115, 3.95e115, 1.7e308, -9e307, 4.5e307, 1e300,
                                     __builtin_huge_val(),
                                     __builtin_nan("")};
constexpr int kSpecial = sizeof special / sizeof special[0];
__device__ double number(unsigned hi, unsigned lo, int emin, int span) {
  const unsigned e = emin + (hi >> 21) % (unsigned)span;   // (the top bit signs)
  return __hiloint2double((int)((hi & 0x800fffffu) | (e << 20)), (int)lo);
}
__global__ void check(int set, unsigned long long* bad) {
  const unsigned i = blockIdx.x * blockDim.x + threadIdx.x;
  double a, b;
  if (set == 2) {
    if (i >= kSpecial * kSpecial) return;
    a = special[i / kSpecial], b = special[i % kSpecial];
  } else {
    unsigned c[4] = {i, (unsigned)set, 0u, 0u};
    philox4x32_10(c, 7u, 11u);
    a = number(c[0], c[1], set ? 0 : 640, set ? 2047 : 767);
    b = number(c[2], c[3], set ? 0 : 640, set ? 2047 : 767);
  }
  if (set == 0) {   // the coarse reciprocal is as good as the derivation takes it to be
    double r;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(b));
    if (!(fabs(fma(-b, r, 1.0)) < 0x1p-19)) atomicAdd(bad, 1ull);
  }
  const double q = quotient(a, b), w = a / b;
  const bool same = __double_as_longlong(q) == __double_as_longlong(w) || (q != q && w != w);
  if (!same && atomicAdd(bad, 1ull) < 8) printf("set %d: %.17g / %.17g = %.17g, not %.17g\n", set, a, b, w, q);
}
int main() {
  unsigned long long *bad, n = 0;
  cudaMalloc(&bad, 8);
  cudaMemset(bad, 0, 8);
  for (int set = 0; set < 3; ++set) check<<<set < 2 ? 65536 : 2, 256>>>(set, bad);
  const bool ok = cudaMemcpy(&n, bad, 8, cudaMemcpyDeviceToHost) == cudaSuccess;
  printf("%s, %llu differ\n", ok ? "done" : "failed", n);
  return ok && n == 0 ? 0 : 1;
}
'''


PAIRS = r'''
#include <cstdio>
#include <cstring>
#include "nmc_internal.cuh"
using namespace nmc;
__device__ df2 number(unsigned hi, unsigned lo, int emin, int span) {   // |low part| <= half a unit of the high one
  const float h = __uint_as_float((hi & 0x807fffffu) | ((unsigned)(emin + (lo & 0xffffu) % (unsigned)span) << 23));
  const float ulp = __uint_as_float((__float_as_uint(h) & 0x7f800000u)) * 0x1p-24f;
  return df_norm(h, ulp * ((float)(int)(lo & 0xffff8000u) * 0x1p-31f));
}
__global__ void check(int set, unsigned long long* bad, unsigned* worst) {
  unsigned c[4] = {blockIdx.x * blockDim.x + threadIdx.x, (unsigned)set, 0u, 1u};
  philox4x32_10(c, 7u, 11u);
  const df2 a = number(c[0], c[1], set ? 200 : 67, set ? 40 : 120);
  const df2 b = number(c[2], c[3], set ? 253 : 67, set ? 2 : 120);
  const double w = df_to_double(a) / df_to_double(b), q = df_to_double(df_div(a, b));
  const double off = fmax(fabs(q - w) - 4 * 0x1p-150, 0.0) / fabs(w);
  if (!set) atomicMax(worst, __float_as_uint((float)off));
  if (!(off <= (set ? 0x1p-20 : 2.75 * 0x1p-46 + 0x1p-53)) && atomicAdd(bad, 1ull) < 8)
    printf("set %d: %.17g / %.17g off by %.3g\n", set, df_to_double(a), df_to_double(b), off);
}
int main() {
  unsigned long long *bad, n = 0;
  unsigned w = 0;
  cudaMalloc(&bad, 16);
  cudaMemset(bad, 0, 16);
  for (int set = 0; set < 2; ++set) check<<<65536, 256>>>(set, bad, (unsigned*)(bad + 1));
  const bool ok = cudaMemcpy(&n, bad, 8, cudaMemcpyDeviceToHost) == cudaSuccess &&
                  cudaMemcpy(&w, bad + 1, 4, cudaMemcpyDeviceToHost) == cudaSuccess;
  float f;
  memcpy(&f, &w, 4);
  printf("%s, %llu off, at most %.3g\n", ok ? "done" : "failed", n, f);
  return ok && n == 0 ? 0 : 1;
}
'''


@pytest.mark.parametrize("program", [PROGRAM, PAIRS], ids=["fp64", "pairs"])
def test_quotients(tmp_path, program):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2106_00712_gb300 import build_lib
    nvcc = build_lib._nvcc()
    assert shutil.which(nvcc), nvcc
    src, exe = tmp_path / "quotients.cu", tmp_path / "quotients"
    src.write_text(program)
    subprocess.run([nvcc, str(src), "-o", str(exe), "-I", build_lib.CSRC] + build_lib.ARCH
                   + build_lib.NVCC_FLAGS, check=True, timeout=300)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
