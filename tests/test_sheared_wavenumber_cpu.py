"""s q_x of the FP32 column passes is the product in double, rounded once
(shf.h: sheared-wavenumber phase in double).  Some of the listed modes lie so
close to a tie that a product of float pairs rounds the other way.  The function
that the kernels call is compiled for the host and compared in bits."""
import math
import subprocess

import numpy as np

from paper_0710_5912_gb300 import _native

# nx, dx, s, modes on both sides of the ties
CASES = [(2048, 1.2392394917709901, -0.85350004550106062, (190, 191, 382, 764, 1023)),
         (4096, 1.0, -0.026449168287097091, (1, 143, 286, 572, 1144, 2047)),
         (4096, 1.3222216175723711, -0.91683742492052644, (0, 531, 1062)),
         (1024, 1.0 / 512, 0.7310585786300049, (1, 77, 511)), (16, 3.7, 127.99, (0, 1, 7))]

SOURCE = """
#include <cstdio>
#include "shf_internal.cuh"
int main() {
  int m; double q, s;
  while (std::scanf("%d %la %la", &m, &q, &s) == 3) {
    float qx, sqx;
    shf::sheared_qx(m, q, s, qx, sqx);
    std::printf("%a %a\\n", qx, sqx);
  }
}
"""


def test_phase_is_the_double_product_rounded_once(tmp_path):
    src, exe = tmp_path / "q.cu", tmp_path / "q"
    src.write_text(SOURCE)
    subprocess.run([_native.nvcc_path(), *_native.ARCH_FLAGS, "-std=c++17", "-O2", "-I", _native.CSRC, "-I",
                    _native.INCLUDE, "-o", str(exe), str(src)], check=True)
    modes = [(m, 2.0 * math.pi / (nx * dx), s) for nx, dx, s, ms in CASES for m in ms]
    out = subprocess.run([str(exe)], input="\n".join(f"{m} {q.hex()} {s.hex()}" for m, q, s in modes), text=True,
                         check=True, stdout=subprocess.PIPE).stdout.split()
    got = np.array([float.fromhex(v) for v in out]).reshape(-1, 2)
    want = np.array([(np.float32(m * q), np.float32(s * (m * q))) for m, q, s in modes], dtype=np.float64)
    assert np.array_equal(got, want)
