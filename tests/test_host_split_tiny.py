"""The FP64 -> pair split below its full-precision range: zeros keep their sign,
magnitudes down to 2^-126 keep the high part's 24 bits, and nothing comes out
larger than it went in (dfloat.cuh, d2df)."""
import math
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tiny_values(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("g++ not available")
    exe = str(tmp_path / "dfh")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_2103_01874_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "dfloat_harness.cpp"), "-o", exe], check=True)
    xs = [s * m * 2.0 ** e for e in (-60, -73, -74, -75, -100, -125, -126, -127, -140, -300, -1000)
          for m in (1.0, 1.7 + 2.0 ** -50, 2.0 - 2.0 ** -52) for s in (1, -1)] + [0.0, -0.0, 5e-324]
    out = subprocess.run([exe], input="\n".join(f"d2df {x.hex()}" for x in xs) + "\n", capture_output=True,
                         text=True, check=True).stdout.split("\n")
    for x, line in zip(xs, out):
        hi, lo = (float.fromhex(t) for t in line.split())
        assert abs(hi) <= max(abs(x), 2.0 ** -126) and abs(lo) <= 2.0 ** -23 * max(abs(hi), 2.0 ** -126)
        if abs(x) >= 2.0 ** -126:
            assert abs(hi + lo - x) <= max(2.0 ** -48 * abs(x), 2.0 ** -149)
        else:
            assert abs(hi + lo) <= 2.0 ** -126
        if x == 0.0:
            assert hi == 0.0 and lo == 0.0 and math.copysign(1, hi) == math.copysign(1, x)
