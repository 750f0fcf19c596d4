"""The FP64 <-> FP32 / double-float / FP16 / BF16 conversions on integer bits give the plain conversions' bits:
every exponent and both ends of the fast ranges, ties, carries into the exponent, zeros,
subnormals, infinities and NaN. The same __host__ __device__ code that the kernels run, in a host
program."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1112_5280_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include "convert.cuh"
using namespace lqcd::cv;
template <class T>
static bool same(T a, T b) {
  return (std::isnan(a) && std::isnan(b)) || !std::memcmp(&a, &b, sizeof a);
}
int main() {
  std::mt19937_64 g(1);
  long long n = 0, bad = 0;
  auto check = [&](double x) {
    ++n;
    volatile float f = (float)x, h = (float)x, l = (float)(x - (double)h);
    bad += !same(to_float(x), (float)f);
    float hi, lo;
    to_df(x, hi, lo);
    bad += !same(hi, (float)h) || !same(lo, (float)l);
    bad += !same(to_double(hi), (double)hi);
    bad += to_half(x) != __half_as_ushort(__double2half(x)) || to_bf16(x) != __bfloat16_as_ushort(__double2bfloat16(x));
    for (float other : {lo, -lo, 0.5f * lo, 3.0f * lo, 0.0f, -0.0f}) bad += !same(from_df(hi, other), (double)hi + (double)other);
  };
  const unsigned long long patterns[] = {0ull, 0x1fffffffull, 0x10000000ull, 0x10000001ull, 0x0fffffffull, 0x20000000ull,
                                         0x30000000ull, 0xfffffe0000000ull, 0xfffffffffffffull, 0xffffff0000000ull,
                                         // ties of FP16 and BF16, next to them, their carries
                                         0x0020000000000ull, 0x0060000000000ull, 0x0020000000001ull, 0x001ffffffffffull,
                                         0xffe0000000000ull, 0x0100000000000ull, 0x0300000000000ull, 0x0100000000001ull,
                                         0x00fffffffffffull, 0xff00000000000ull};
  for (unsigned long long sign : {0ull, 1ull << 63})
    for (unsigned long long e = 0; e < 2048; ++e) {
      for (int k = 0; k < 1000; ++k) {
        unsigned long long m = k < 20 ? patterns[k] : g() & 0xfffffffffffffull;
        if (k >= 20 && k % 3 == 0) m = (m & ~0x1fffffffull) | patterns[k % 7];
        if (k >= 20 && k % 3 == 1) m = (m & ~0x3ffffffffffull) | patterns[10 + k % 4];
        const unsigned long long b = sign | (e << 52) | m;
        double x;
        std::memcpy(&x, &b, 8);
        check(x);
      }
    }
  std::printf("%lld %lld\n", n, bad);
  return bad != 0;
}
"""


def _nvcc():
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else shutil.which("nvcc")


def test_conversions_equal_the_plain_ones(tmp_path):
    nvcc = _nvcc()
    if not nvcc:
        pytest.skip("nvcc not available")
    src = tmp_path / "convert.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "convert"
    subprocess.run([nvcc, "-std=c++17", "-O2", "-Wno-deprecated-gpu-targets", f"-I{CSRC}",
                    f"-I{os.path.join(ROOT, 'include')}", "-o", str(exe), str(src)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.split() == [str(2 * 2048 * 1000), "0"]
