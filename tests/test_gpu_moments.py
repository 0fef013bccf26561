"""The additions of the structure factor's moments are compensated down to a
thread's own modes.  On one 16 x 16 CTA a wave of period 4 and a point make one
mode of S = 2 and 118 modes of a fraction of its last place, all computed
exactly (the transform meets no twiddle factor but quarter turns); seven of the
small modes share the large one's thread.  Added without compensation two of
these are lost and four round away from their sum (1.2 units of the last place).
The result may be half a unit off (its own rounding)."""
import math
from fractions import Fraction

import numpy as np
import pytest

import paper_0710_5912_gb300 as shf

pytestmark = pytest.mark.gpu


def test_small_modes_beside_a_large_one_are_kept():
    n = 16
    e = 641316 / 2 ** 20 * 2.0 ** -18                   # e^2 / 2^15 = 0.374 units of the last place of 2
    phi = np.tile(np.array([1.0, 0.0, -1.0, 0.0]) * ((256.0 - e) / 128.0), (n, n // 4))
    phi[0, 0] += e
    with shf.Grid(n, n, 1.0, shf.SHF_FP64) as g:
        g.set_params()
        g.set_fields(phi)
        moments, _ = g.structure_factor()
        tensor, _ = g.gradient_tensor()
    unit = Fraction(1, 2 ** 51)
    small = Fraction(2 * (e / 256.0) ** 2)              # (rounded as the kernel's)
    want = 2 + 104 * small + 14 * small / 2             # columns 1..7 off the Nyquist row, and column 0 off k = 0
    assert abs(Fraction(moments[0]) - want) <= Fraction(3, 4) * unit
    # sum q_x^2 S / sum S, k = 0 included below: q_x^2, the sum and the quotient round
    q = [2.0 * math.pi * m / n for m in range(8)]
    num = 2 * Fraction(q[4] * q[4]) + sum((14 if m == 4 else 15) * small * Fraction(q[m] * q[m]) for m in range(1, 8))
    G = num / (want + small / 2)
    assert abs(Fraction(tensor[0]) / G - 1) <= Fraction(3, 2 ** 53)
