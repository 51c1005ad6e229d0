"""The per-gate kernels' binary64 <-> double-float conversions against the tile kernels', bit for bit, on
the host: ordinary values, both ends of the float range, powers of two, zeros and short mantissas."""
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2010_09746_gb300", "csrc")

SRC = r"""
#include <cstdio>
#include <cstring>
#include <random>
#include "arith.cuh"
using namespace qs;
int main() {
  std::mt19937_64 g(1);
  long bad = 0;
  for (long i = 0; i < 4000000; i++) {
    unsigned long long b = g();
    const int kind = (int)(i % 4);
    const int e = kind == 0 ? 1023 - (int)(g() % 60) : kind == 1 ? 880 + (int)(g() % 150) : kind == 2 ? (int)(g() % 1151)
                                                                                                     : 1023 + (int)(g() % 100);
    b = (b & 0x800fffffffffffffull) | ((unsigned long long)e << 52);
    if (i % 7 == 0) b &= ~((1ull << (g() % 53)) - 1);
    if (i % 1001 == 0) b &= 0x8000000000000000ull;
    double x;
    memcpy(&x, &b, 8);
    const dfl o = split_double(x), n = split_double_gate(x);
    bad += memcmp(&o, &n, 8) != 0;
    float h = o.hi, l = o.lo;
    if (i % 5 == 0) l = -l;
    if (i % 11 == 0) l = 0;
    if (i % 13 == 0) l = h * ldexpf((float)((g() % 2001) / 1000.0 - 1), -24 - (int)(g() % 30));
    if (i % 17 == 0) h = f_from_bits(f_bits(h) & 0xff800000u);   // a power of two
    const dfl q = two_sum(h, l);
    const double a = join_double(q.hi, q.lo), c = join_double_gate(q.hi, q.lo);
    bad += memcmp(&a, &c, 8) != 0;
  }
  printf("%ld\n", bad);
}
"""


def test_same_bits(tmp_path):
    nvcc = next((c for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", shutil.which("nvcc")) if c and os.path.exists(c)),
                None)
    if nvcc is None:
        pytest.skip("nvcc not available")
    src, exe = tmp_path / "convert.cu", tmp_path / "convert"
    src.write_text(SRC)
    r = subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-std=c++17", "-O2", "-Xcompiler", "-ffp-contract=off",
                        "-I", CSRC, "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout.strip() == "0"
