"""How often the integer-pipe power of two (csrc/pow2_fixed.cuh, compiled for the
host) is not the nearest float64.

Before its rounding to 53 bits the result is off by at most 2^-60.  An error of
delta 2^-60 misrounds a share of about delta 2^-7 (half of it for mantissas near 2) of
all results.  Its mean is 0.12 2^-60 and its spread 0.17 2^-60: with the mean taken
out by the rounding constant the mean of |delta| is 0.13 and the share at most 1e-3 of
mantissas at 1, about 7e-4 of all; with the mean left in it is 1.3e-3.  Asserted below
9e-4 over 120,000 arguments (a standard deviation of 8e-5).
"""
import os
import struct
import subprocess

import numpy as np
from mpmath import mp, mpf

HERE = os.path.dirname(os.path.abspath(__file__))
HDR = os.path.join(os.path.dirname(HERE), "paper_2305_18025_gb300", "csrc", "pow2_fixed.cuh")
DRIVER = r"""
#include <cstdio>
#include "%s"
int main() {
  unsigned long long b;
  while (std::scanf("%%llx", &b) == 1) {
    const bpimd::pow2fx::mexp r = bpimd::pow2fx::pow2neg(bpimd::pow2fx::bits_to_double(b), bpimd::pow2fx::T63);
    std::printf("%%llx %%d\n", bpimd::pow2fx::double_to_bits(r.m), r.e);
  }
  return 0;
}
"""


def test_share_of_misrounded_results(tmp_path):
    src, exe = tmp_path / "d.cpp", tmp_path / "d"
    src.write_text(DRIVER % HDR)
    subprocess.run(["g++", "-O2", "-std=c++17", "-o", str(exe), str(src)], check=True)
    x = np.random.default_rng(4).uniform(0.0, 40.0, 120000)
    lines = "\n".join("%x" % struct.unpack("<Q", struct.pack("<d", v))[0] for v in x)
    out = subprocess.run([str(exe)], input=lines + "\n", capture_output=True, text=True, check=True).stdout.split()
    mp.prec = 120
    wrong = 0
    for v, m, e in zip(x, out[::2], out[1::2]):
        m53 = (int(m, 16) & ((1 << 52) - 1)) | (1 << 52)
        exact = mp.power(2, -mpf(float(v)) - int(e) + 52)
        wrong += abs(exact - m53) > mpf(0.5) * (1 + mpf(2) ** -60)
    assert wrong < 9e-4 * len(x), wrong / len(x)
