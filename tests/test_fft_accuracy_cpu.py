"""Rounding of the double-precision register FFT against long double.  The
limits are the errors on the same inputs of a transform with separate factors (a
radix-8 DFT of additions whose inputs are multiplied by products of two table
entries): butterflies with fused factors save instructions, not digits."""
import os
import shutil
import subprocess

import pytest

from paper_0710_5912_gb300 import _native

LIMITS = {16: 1.215e-16, 32: 1.364e-16, 64: 1.809e-16, 128: 1.911e-16, 256: 2.034e-16, 512: 2.351e-16, 1024: 2.490e-16}


def test_fused_factors_round_no_worse_than_separate_ones(tmp_path):
    if shutil.which("g++") is None:
        pytest.skip("no host compiler")
    here = os.path.dirname(os.path.abspath(__file__))
    cuda = os.path.join(os.path.dirname(os.path.dirname(_native.nvcc_path())), "include")
    exe = str(tmp_path / "fft")
    subprocess.run(["g++", "-std=c++20", "-O2", "-w", "-pthread", "-I", cuda, "-I", _native.CSRC, "-o", exe,
                    os.path.join(here, "fft_accuracy.cpp")], check=True)
    out = subprocess.run([exe], check=True, text=True, stdout=subprocess.PIPE).stdout
    for line in out.splitlines():
        n, fwd, inv = line.split()
        assert max(float(fwd), float(inv)) <= LIMITS[int(n)], line
    assert len(out.splitlines()) == len(LIMITS)
